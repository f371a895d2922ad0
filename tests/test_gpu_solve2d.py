"""The one-launch 2D solve: its sums of products against exact sums, and the range
of right-hand sides, box sizes and starts that it takes."""
import ctypes
import math
import subprocess

import numpy as np
import pytest

import pf_inputs as I
from oracle import pf_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g

    g.build()
    import paper_2205_05835_gb300 as pf

    return pf


SUMS = r"""
#include "pf_solve2d.cuh"
using A = pf::S2AccOf<float>::type;
// thread t: n products; thread 0 then merges the block's accumulators
__global__ void k_sums(const float* a, const float* b, int n, double* out) {
    __shared__ A all[64];
    A v{};
    for (int i = 0; i < n; ++i) v.add_prod(a[threadIdx.x * n + i], b[threadIdx.x * n + i]);
    all[threadIdx.x] = v;
    out[threadIdx.x] = v.value();
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int t = 1; t < 64; ++t) v.merge(all[t]);
        out[64] = v.value();
    }
}
extern "C" int run(const float* a, const float* b, int n, double* out) {
    k_sums<<<1, 64>>>(a, b, n, out);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.mark.parametrize("n", [1, 2, 7, 32, 200])
def test_sums_of_products_are_as_accurate_as_float64_ones(pf, tmp_path, n):
    """The mixed path's accumulators on 64 threads of n products, built with the
    library's flags: random products, and ones that cancel to 2^-20 of their
    size. The float64 sums that they stand for are off by at most 2^-53 sum|a b|
    for every addition."""
    import torch

    from paper_2205_05835_gb300 import build as B

    src, lib = tmp_path / "sums.cu", tmp_path / "sums.so"
    src.write_text(SUMS)
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC, "-shared", "-o", str(lib), str(src)],
                   check=True, capture_output=True)
    run = ctypes.CDLL(str(lib)).run
    rng = np.random.default_rng(n)
    a = rng.standard_normal((64, n)).astype(np.float32)
    b = rng.standard_normal((64, n)).astype(np.float32)
    cancel = a.copy()
    cancel[:, n // 2:2 * (n // 2)] = -a[:, :n // 2] * np.float32(1 + 2.0 ** -20)
    bc = b.copy()
    bc[:, n // 2:2 * (n // 2)] = b[:, :n // 2]
    for x, y in ((a, b), (cancel, bc)):
        dx, dy = torch.tensor(x, device="cuda"), torch.tensor(y, device="cuda")
        out = torch.zeros(65, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert run(ctypes.c_void_p(dx.data_ptr()), ctypes.c_void_p(dy.data_ptr()), n,
                   ctypes.c_void_p(out.data_ptr())) == 0
        got = out.cpu().numpy()
        prod = x.astype(np.float64) * y.astype(np.float64)   # exact: 24 + 24 bits
        want = np.array([math.fsum(r) for r in prod] + [math.fsum(prod.reshape(-1))])
        size = np.append(np.abs(prod).sum(axis=1), np.abs(prod).sum())
        count = np.append(np.full(64, n), 64 * n)
        assert (np.abs(got - want) <= 2.0 ** -53 * count * size).all()


def beta32(phi, g, p):
    """The mixed path's float32 face coefficients, operation by operation."""
    f = np.float32
    c = np.clip(phi.astype(f), f(0), f(1))
    rho = f(p["rho_out"]) + (f(p["rho_in"]) - f(p["rho_out"])) * c
    return [(f(1) / (f(0.5) * (rho + np.roll(rho, 1, g.axis(d))))).astype(np.float64)
            for d in range(2)]


def mixed_solve(pf, n, L, ratio, rhs, x0=None):
    """(status, iterations, relative residual formed here in float64)."""
    p = I.small_case(dim=2, n=n, precision="mixed", poisson_rtol=1e-10, L=L, R=0.25 * L,
                     rho_in=10.0, rho_out=10.0 / ratio)
    po = O.params_from(p)
    g = O.Grid(2, (n, n), L)
    phi = O.initial_phi(po).astype(np.float32).astype(np.float64)
    sim = pf.Simulation(p, phi0=phi)
    x, iters, rel, status = sim.poisson_solve(rhs, x0)
    sim.close()
    r = rhs - rhs.mean() - O.apply_poisson(beta32(phi, g, p), x, g)
    return status, iters, np.linalg.norm(r) / np.linalg.norm(rhs - rhs.mean())


@pytest.mark.parametrize("n", [64, 256])
@pytest.mark.parametrize("amp", [1e-25, 1e-20, 1e-12, 1e-9, 1e6, 1e12, 1e20, 1e30])
def test_mixed_solve_takes_any_amplitude(pf, n, amp):
    """The solve is linear in its right-hand side, so its size changes neither the
    convergence nor (by more than the test's own rounding) the residual. The
    bound is rtol, plus the rounding of x as the double-float that holds it
    (2^-46 and, in its low word, float's smallest number) through the operator."""
    noise = I.noise((n, n), 6) - 0.5
    st1, it1, rel1 = mixed_solve(pf, n, 1.0, 10.0, noise)
    st, it, rel = mixed_solve(pf, n, 1.0, 10.0, amp * noise)
    assert st1 == 0 and rel1 <= 1.1e-10
    assert st == 0 and abs(it - it1) <= 1
    assert rel <= 1.1e-10 + 8.0 * n * n * 2.0 ** -149 / (0.28 * amp)


@pytest.mark.parametrize("L,amp", [(1e-6, 1.0), (1e-2, 1e-8), (1e-2, 1e8), (1e3, 1.0)])
def test_mixed_solve_takes_any_box(pf, L, amp):
    noise = I.noise((64, 64), 6) - 0.5
    st1, it1, _ = mixed_solve(pf, 64, 1.0, 10.0, noise)
    st, it, rel = mixed_solve(pf, 64, L, 10.0, amp * noise)
    assert st1 == 0 and st == 0 and abs(it - it1) <= 1
    assert rel <= 1.1e-10


@pytest.mark.parametrize("ratio", [10.0, 1000.0])
@pytest.mark.parametrize("start", [1e6, 1e13])
def test_mixed_solve_takes_any_start(pf, ratio, start):
    """A start whose residual is beyond float32's squares is worked off. (A constant
    of at most its size stays in x meanwhile, and with it the rounding of a double-
    float, 2^-47 of it times the operator's 8 max beta / h^2, so a first call may stop
    short; x is returned with zero mean.)"""
    rhs = I.noise((64, 64), 6) - 0.5
    p = I.small_case(dim=2, n=64, precision="mixed", poisson_rtol=1e-10, rho_in=10.0,
                     rho_out=10.0 / ratio)
    sim = pf.Simulation(p)
    x, _, rel, status = sim.poisson_solve(rhs, start * (I.noise((64, 64), 7) - 0.5))
    floor = 2.0 ** -47 * start * 8.0 * max(0.1, 0.1 * ratio) * 64 ** 2 / 0.28
    assert status in (pf.B.PF_OK, pf.B.PF_ERR_NOT_CONVERGED) and rel <= 1e-10 + floor
    x, _, rel, status = sim.poisson_solve(rhs, x)
    assert status == pf.B.PF_OK and rel <= 1e-10
    sim.close()


def test_mixed_solve_of_zero_and_of_a_nan(pf):
    zero = np.zeros((64, 64))
    p = I.small_case(dim=2, n=64, precision="mixed", poisson_rtol=1e-10)
    sim = pf.Simulation(p)
    x, iters, rel, status = sim.poisson_solve(zero)
    assert status == 0 and iters == 0 and not x.any()
    bad = I.noise((64, 64), 6)
    bad[3, 5] = np.nan
    with pytest.raises(pf.PFError) as e:
        sim.poisson_solve(bad)
    assert e.value.status == pf.B.PF_ERR_NONFINITE
    x, iters, rel, status = sim.poisson_solve(I.noise((64, 64), 6) - 0.5)
    assert status == 0 and rel <= 1e-10
    sim.close()


# tolerances between the residuals at which rounding stops the two solves (64
# refinements): measured 9.6e-12 and at most 3.1e-12 at 256^2, 6.2e-11 and at most 3.1e-12 at
# 640^2 (beyond the one-launch solve), 5.3e-13 and at most 8.2e-14 at 64^3
@pytest.mark.parametrize("n,rtol", [((256, 256), 6e-12), ((640, 640), 2e-11),
                                    ((64, 64, 64), 2e-13)])
def test_graph_reports_a_solve_that_stops_at_the_refinement_limit(pf, n, rtol):
    """Two forward-Euler steps of one call in graph mode, at density ratio 1 from a
    smooth potential flow. The first solve's pressure is large against its right-
    hand side, so its rounding keeps it above rtol; the second's right-hand side
    is what the projection left, which is rough, and converges. The first one's
    failure is reported."""
    p = I.small_case(dim=len(n), n=n[0], precision="mixed", poisson_rtol=rtol, rho_in=1.0,
                     rho_out=1.0, sigma=0.0, mu_in=0.0, mu_out=0.0, scheme="fe",
                     poisson_maxit=5000, use_graph=1, pert_mode=0, pert_amp=0.0)
    t = 2.0 * np.pi * np.arange(n[0]) / n[0]
    tc = t + np.pi / n[0]
    u = (1.0 + 0.5 * np.cos(tc + 1.1))[:, None] * np.sin(t + 0.3)[None, :]
    v = 0.5 * np.sin(t + 1.1)[:, None] * np.cos(tc + 0.3)[None, :]

    def fresh():
        sim = pf.Simulation(p)
        sim.set_field("u", np.broadcast_to(u, sim.shape))
        sim.set_field("v", np.broadcast_to(v, sim.shape))
        return sim

    sim = fresh()
    with pytest.raises(pf.PFError) as e:
        sim.step(1)
    assert e.value.status == pf.B.PF_ERR_NOT_CONVERGED
    sim.step(1)   # the second step's solve converges, and the latch is clear
    sim.close()
    sim = fresh()
    with pytest.raises(pf.PFError) as e:
        sim.step(2)
    assert e.value.status == pf.B.PF_ERR_NOT_CONVERGED
    sim.close()


# the last three: the next split's strip is too large, or none fits
@pytest.mark.parametrize("n,precision,cluster",
                         [((64, 64), "fp64", True), ((512, 512), "fp64", True),
                          ((268, 268), "fp64", True), ((512, 40), "fp64", True),
                          ((300, 300), "fp64", True), ((468, 156), "fp64", True),
                          ((313, 54), "fp64", True), ((468, 276), "mixed", True),
                          ((512, 512), "mixed", True), ((548, 164), "fp64", False),
                          ((580, 276), "mixed", False), ((1000, 200), "fp64", False)])
def test_which_solve_a_grid_takes(pf, n, precision, cluster):
    rtol = 1e-11 if precision == "fp64" else 1e-10
    p = I.small_case(dim=2, n=n[0], precision=precision, poisson_rtol=rtol,
                     R=0.25 * min(1.0, n[1] / n[0]))
    p["n"] = n + (1,)
    po = O.params_from(p)
    g = O.Grid(2, n, p["L"])
    phi = O.initial_phi(po).astype(np.float32).astype(np.float64)
    rhs = I.noise(g.shape, 6) - 0.5
    rhs -= rhs.mean()
    sim = pf.Simulation(p, phi0=phi)
    x, iters, rel, status = sim.poisson_solve(rhs)
    ran = pf.pf_profile_read(sim.ctx)
    sim.close()
    assert (ran.get("solve2d_cluster", (0, 0.0))[0] > 0) == cluster
    assert (ran.get("cg_update", (0, 0.0))[0] > 0) != cluster
    beta = O.face_beta(phi, g, po) if precision == "fp64" else beta32(phi, g, p)
    r = rhs - O.apply_poisson(beta, x, g)
    # rounding of x (2^-47 for a double-float, 2^-52 for float64) through the operator
    eps = 2.0 ** -47 if precision == "mixed" else 2.0 ** -52
    floor = 8.0 * eps * max(b.max() for b in beta) / g.h ** 2 * np.linalg.norm(x)
    assert status == 0 and iters <= 40
    assert np.linalg.norm(r) <= 1.01 * rtol * np.linalg.norm(rhs) + floor

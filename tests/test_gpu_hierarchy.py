"""Pressure solves on grids whose multigrid hierarchy has odd sizes, short axes
or unequal axes, against the oracle's exact solve of the same operator."""
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


def beta32(phi, g, p):
    """The mixed path's float32 face coefficients, operation by operation."""
    f = np.float32
    c = np.clip(phi.astype(f), f(0), f(1))
    rho = f(p["rho_out"]) + (f(p["rho_in"]) - f(p["rho_out"])) * c
    return [(f(1) / (f(0.5) * (rho + np.roll(rho, 1, g.axis(d))))).astype(np.float64)
            for d in range(g.dim)]


SIZES = [(4, 4), (5, 4), (7, 63), (33, 31), (61, 45), (64, 64), (100, 36), (200, 6), (130, 66),
         (6, 5, 4), (9, 7, 5), (20, 15, 9), (24, 4, 50), (17, 18, 13), (32, 20, 12)]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_solve_on_any_size(pf, n, precision):
    rtol = 1e-11 if precision == "fp64" else 1e-9
    p = I.small_case(dim=len(n), n=n[0], precision=precision, poisson_rtol=rtol, R=0.2)
    p["n"] = tuple(n) + (1,) * (3 - len(n))
    p = I.finalize(p)
    po = O.params_from(p)
    g = O.Grid(len(n), n, p["L"])
    phi = np.clip(O.initial_phi(po) + 0.1 * (I.noise(g.shape, 5) - 0.5), 0.0, 1.0)
    phi = phi.astype(np.float32).astype(np.float64)
    rhs = I.noise(g.shape, 6) - 0.5
    sim = pf.Simulation(p, phi0=phi)
    x, iters, rel, status = sim.poisson_solve(rhs)
    sim.close()
    beta = O.face_beta(phi, g, po) if precision == "fp64" else beta32(phi, g, p)
    want = O.solve_poisson(beta, rhs, g)
    assert status == 0 and rel <= rtol
    # |x - x*| <= |r| / lambda_min <= rtol |f| / lambda_min in the 2-norm (plus the
    # rounding of the double-float right-hand side, 2^-47, in the mixed form);
    # lambda_min >= min beta (smallest non-zero eigenvalue of the Laplacian)
    h = g.h
    lam = min(b.min() for b in beta) * (2 - 2 * np.cos(2 * np.pi / max(n))) / h ** 2
    f = rhs - rhs.mean()
    assert np.linalg.norm(x - want) <= (1.01 * rtol + 2.0 ** -40) * np.linalg.norm(f) / lam
    # a V-cycle that halves the error per iteration or better
    assert iters <= np.log2(1.0 / rtol) + 4


@pytest.mark.parametrize("n,ratio", [((64, 64), 1000.0), ((256, 256), 1000.0), ((320, 320), 10.0),
                                     ((512, 40), 10.0), ((384, 512), 10.0), ((512, 512), 10.0),
                                     ((650, 650), 10.0), ((700, 700), 10.0)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("sweeps", [1, 2])
def test_2d_solve_residual(pf, n, ratio, precision, sweeps):
    """Strips of unequal rows, arrays that overflow into the workspace, the
    largest grids of the one-launch solve and the multi-kernel solve beyond it:
    the residual of the returned x, formed here, meets the tolerance."""
    rtol = 1e-10
    p = I.small_case(dim=2, n=n[0], precision=precision, poisson_rtol=rtol, rho_in=10.0,
                     rho_out=10.0 / ratio, mg_pre=sweeps, mg_post=sweeps)
    p["n"] = n + (1,)
    p = I.finalize(p)
    po = O.params_from(p)
    g = O.Grid(2, n, p["L"])
    phi = O.initial_phi(po).astype(np.float32).astype(np.float64)
    rhs = I.noise(g.shape, 6) - 0.5
    rhs -= rhs.mean()
    sim = pf.Simulation(p, phi0=phi)
    x, iters, rel, status = sim.poisson_solve(rhs)
    sim.close()
    beta = O.face_beta(phi, g, po) if precision == "fp64" else beta32(phi, g, p)
    r = rhs - O.apply_poisson(beta, x, g)
    # rounding of x (2^-47 for a double-float, 2^-52 for float64) through the operator
    eps = 2.0 ** -47 if precision == "mixed" else 2.0 ** -52
    floor = 8.0 * eps * max(b.max() for b in beta) / g.h ** 2 * np.linalg.norm(x)
    assert status == 0 and iters <= 40
    assert np.linalg.norm(r) <= 1.01 * rtol * np.linalg.norm(rhs) + floor


@pytest.mark.parametrize("n", [(32, 20, 12), (48, 32, 24), (24, 24, 24), (30, 22, 26)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("sweeps", [1, 2, 3])
def test_3d_solve_residual(pf, n, precision, sweeps):
    """The 3D hierarchy with several sweeps a level: the first-colour restriction
    and inverse diagonals of the float64 levels, the cluster kernel below."""
    rtol = 1e-10
    p = I.small_case(dim=3, n=n[0], precision=precision, poisson_rtol=rtol, R=0.2,
                     mg_pre=sweeps, mg_post=sweeps)
    p["n"] = n
    p = I.finalize(p)
    po = O.params_from(p)
    g = O.Grid(3, n, p["L"])
    phi = O.initial_phi(po).astype(np.float32).astype(np.float64)
    rhs = I.noise(g.shape, 6) - 0.5
    rhs -= rhs.mean()
    sim = pf.Simulation(p, phi0=phi)
    x, iters, rel, status = sim.poisson_solve(rhs)
    sim.close()
    beta = O.face_beta(phi, g, po) if precision == "fp64" else beta32(phi, g, p)
    r = rhs - O.apply_poisson(beta, x, g)
    eps = 2.0 ** -47 if precision == "mixed" else 2.0 ** -52
    floor = 12.0 * eps * max(b.max() for b in beta) / g.h ** 2 * np.linalg.norm(x)
    assert status == 0 and iters <= 36
    assert np.linalg.norm(r) <= 1.01 * rtol * np.linalg.norm(rhs) + floor


@pytest.mark.parametrize("n", [(40, 24, 16), (72, 40, 24), (132, 36, 20), (68, 20, 140)])
@pytest.mark.parametrize("ratio", [10.0, 1000.0])
def test_3d_mixed_first_colour_restriction(pf, n, ratio):
    """Column-marching restriction after one sweep from zero (first colour alone,
    from densities and, below level 1, from face arrays), ragged column tiles and
    several z chunks: against the one that reads every cell (two sweeps). A
    V(2, 2) cycle does no more than two V(1, 1) cycles, so one sweep takes at
    most twice its iterations (and one per refinement, of which there are two)."""
    iters = {}
    for sweeps in (1, 2):
        p = I.small_case(dim=3, n=n[0], precision="mixed", poisson_rtol=1e-10, R=0.2,
                         rho_in=10.0, rho_out=10.0 / ratio, mg_pre=sweeps, mg_post=sweeps,
                         mg_coarse_cells=64)
        p["n"] = n
        p = I.finalize(p)
        po = O.params_from(p)
        g = O.Grid(3, n, p["L"])
        phi = O.initial_phi(po).astype(np.float32).astype(np.float64)
        rhs = I.noise(g.shape, 6) - 0.5
        rhs -= rhs.mean()
        sim = pf.Simulation(p, phi0=phi)
        x, iters[sweeps], rel, status = sim.poisson_solve(rhs)
        sim.close()
        beta = beta32(phi, g, p)
        r = rhs - O.apply_poisson(beta, x, g)
        floor = 12.0 * 2.0 ** -47 * max(b.max() for b in beta) / g.h ** 2 * np.linalg.norm(x)
        assert status == 0
        assert np.linalg.norm(r) <= 1.01e-10 * np.linalg.norm(rhs) + floor
    assert iters[1] <= 2 * iters[2] + 2

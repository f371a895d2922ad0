"""The plan of the one-launch 2D solve (which CTAs hold what) on the host: which
grids take it, and that the layout they get is sound."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_05835_gb300", "csrc")

SHIM = r"""
#include "pf_solve2d.cuh"
using namespace pf;
template <typename T>
static int run(int nx, int ny, int ctas, int* out) {
    static MGHier<T> H;
    mg_geometry(H, make_dims(nx, ny, 1, 1.0), 2, false);
    H.pre = H.post = 1;
    const S2Limits lim = s2_limits<T>(ctas, s2_dynamic_smem<T>());
    static S2Plan P, Q;
    const int got = s2_plan<T>(H, lim, true, true, P) ? 1 : 0;
    // of the splits that fit, the cheapest one's largest strip (0: none fits; negative:
    // it is the cheapest of all)
    int strip = 0;
    float least = 1e30f, fitting = 1e30f;
    if (H.lev[H.nlev - 1].g.ncell <= lim.dense_cells)
        for (int lc = 1; lc < H.nlev && lc < kS2MaxCluster; ++lc)
            for (int C = 1; C <= ctas && C <= H.lev[lc].g.ny; C *= 2) {
                for (int l = 0; l < H.nlev; ++l) {
                    Q.lev[l].nx = H.lev[l].g.nx;
                    Q.lev[l].ny = H.lev[l].g.ny;
                    Q.lev[l].qx = H.lev[l].lastw[0];
                    Q.lev[l].qy = H.lev[l].lastw[1];
                }
                Q.lc = lc;
                Q.C = C;
                const float c = s2_cost(Q, H.nlev, lim);
                const bool fit = s2_place(Q, lim, sizeof(T), true, true);
                if (c < least) least = c;
                if (fit && c < fitting) {
                    fitting = c;
                    strip = s2_max_rows(Q, 0) * nx;
                }
            }
    if (strip && fitting == least) strip = -strip;
    int n = 0;
    auto put = [&](int v) { out[n++] = v; };
    put(strip);
    if (!got) return 0;
    put(P.C), put(P.lc), put(P.ld), put(P.elems), put(H.nlev);
    put(P.om), put(P.lev[P.ld].nx * P.lev[P.ld].ny * s2_pad(P.lev[P.ld].nx * P.lev[P.ld].ny));
    for (int l = 0; l <= P.ld; ++l) {
        const S2Lev& L = P.lev[l];
        const int c = s2_max_rows(P, l) * L.nx;
        for (int o : {L.ox, L.of, L.ow0, L.ow1, L.od}) put(o), put(c);
        if (l == 0)
            for (int o : {P.op, P.oq, P.oe, P.os}) put(o), put(c);
    }
    put(-7);
    for (int l = 0; l <= P.lc; ++l) {
        put(H.lev[l].g.ny);
        for (int c = 0; c <= P.C; ++c) put(s2_row(P, l, c));
    }
    return n;
}
extern "C" int plan(int nx, int ny, int f32, int ctas, int* out) {
    return f32 ? run<float>(nx, ny, ctas, out) : run<double>(nx, ny, ctas, out);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("plan")
    (d / "p.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-shared", "-fPIC", "-I", CSRC, "-I", inc,
                    "-o", str(d / "p.so"), str(d / "p.cpp")], check=True, capture_output=True)
    fn = ctypes.CDLL(str(d / "p.so")).plan
    out = (ctypes.c_int * 1024)()

    def call(nx, ny, precision, ctas=16):
        n = fn(nx, ny, int(precision == "mixed"), ctas, out)
        return list(out[:max(n, 1)])

    return call


def check_layout(v):
    """Arrays inside the shared memory, aligned and apart; strips that cover the rows
    in order, none empty, each level's strips on twice the next level's."""
    C, lc, ld, elems = v[1:5]
    end = v.index(-7)
    arrays = [(v[i], v[i + 1]) for i in range(6, end, 2) if v[i] >= 0]
    arrays.sort()
    assert all(o % 4 == 0 for o, _ in arrays)
    assert all(o + c <= p for (o, c), (p, _) in zip(arrays, arrays[1:]))
    assert arrays[-1][0] + arrays[-1][1] <= elems
    rows = np.array(v[end + 1:]).reshape(lc + 1, C + 2)
    ny, r = rows[:, 0], rows[:, 1:]
    assert (r[:, 0] == 0).all() and (r[:, -1] == ny).all() and (np.diff(r, axis=1) > 0).all()
    assert (r[:-1, :-1] == 2 * r[1:, :-1]).all()


@pytest.mark.parametrize("n", [(268, 268), (512, 40), (1024, 64), (468, 156), (300, 300)])
def test_float64_grids_whose_cheapest_split_does_not_fit(plan, n):
    v = plan(*n, "fp64")
    assert v[0] > 0 and len(v) > 1
    check_layout(v)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_a_grid_takes_the_cheapest_split_that_fits(plan, precision):
    """Whatever its strip where no other split is cheaper, else up to the strip at
    which the kernels are faster (half of it on odd sizes)."""
    most = {"fp64": 9500, "mixed": 13500}[precision]
    rng = np.random.default_rng(5)
    sizes = [(a, b) for a in (4, 5, 16, 63, 64, 200, 512, 513) for b in (4, 7, 40, 64, 384, 512)]
    sizes += [tuple(int(x) for x in np.exp(rng.uniform(np.log(4), np.log(1400), 2)))
              for _ in range(3000)]
    taken = 0
    for nx, ny in sizes:
        for ctas in (16, 8):
            v = plan(nx, ny, precision, ctas)
            take = v[0] < 0 or 0 < v[0] <= (most // 2 if (nx | ny) & 1 else most)
            assert (len(v) > 1) == take, (nx, ny, ctas)
            if len(v) > 1:
                assert v[4] * (4 if precision == "mixed" else 8) <= 227 * 1024
                check_layout(v)
                taken += 1
    assert taken > 1000


@pytest.mark.parametrize("n", [(1024, 1024), (600, 600), (66000, 4)])
def test_large_grids_do_not_take_it(plan, n):
    assert len(plan(*n, "mixed")) == 1 and len(plan(*n, "fp64")) == 1

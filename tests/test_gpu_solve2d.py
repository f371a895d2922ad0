"""The one-launch 2D solve: its sums of products against exact sums."""
import ctypes
import math
import subprocess

import numpy as np
import pytest

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

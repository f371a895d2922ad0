"""The planes per CTA of the kernels that march in z, on the host: the rule's choice
against measured times."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_05835_gb300", "csrc")

# outer residual of the 3D mixed solve on a GB300, us a launch by the number of chunks
MEASURED = {
    (192, 192, 192): {24: 98.1, 16: 95.7, 12: 94.0, 9: 98.1, 8: 104.3, 7: 109.6, 6: 88.2,
                      5: 98.2, 4: 102.7, 3: 124.7},
    (224, 224, 224): {28: 147.2, 19: 137.4, 14: 142.2, 11: 142.1, 10: 129.0, 8: 136.1, 7: 141.6,
                      6: 156.0, 5: 158.8, 4: 144.5},
    (256, 256, 256): {32: 207.7, 22: 194.0, 16: 190.0, 12: 189.2, 11: 187.7, 10: 187.8, 8: 196.8,
                      7: 176.8, 6: 189.3, 5: 216.6, 4: 239.5},
    (320, 320, 320): {40: 389.2, 27: 357.6, 20: 349.2, 15: 333.5, 14: 334.5, 12: 328.3, 10: 338.8,
                      9: 325.9, 8: 339.4, 7: 344.9, 6: 341.3, 5: 368.5},
    (512, 512, 64): {8: 209.3, 6: 193.3, 4: 191.5, 3: 183.4, 2: 183.4, 1: 241.3},
    (128, 128, 128): {16: 41.6, 11: 36.7, 8: 40.2, 6: 45.1, 5: 52.3, 4: 57.3, 3: 71.4, 2: 98.3},
}


@pytest.fixture(scope="module")
def march_zc(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("march")
    (d / "m.cpp").write_text('#include "pf_internal.h"\n'
                             'extern "C" int zc(long long cols, int nz, long long slots, int extra)'
                             ' { return pf::march_zc(cols, nz, slots, extra); }\n')
    subprocess.run(["g++", "-std=c++17", "-w", "-shared", "-fPIC", "-I", CSRC, "-I", inc, "-o",
                    str(d / "m.so"), str(d / "m.cpp")], check=True, capture_output=True)
    fn = ctypes.CDLL(str(d / "m.so")).zc
    fn.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_longlong, ctypes.c_int]
    return fn


@pytest.mark.parametrize("n", list(MEASURED))
def test_the_residuals_chunk_is_near_the_best_measured_one(march_zc, n):
    """Six CTAs resident per SM; a number of chunks between two measured ones counts as
    the slower of them."""
    cols = ((n[0] + 31) // 32) * ((n[1] + 7) // 8)
    zc = march_zc(cols, n[2], 6 * 152, 6)
    chunks = (n[2] + zc - 1) // zc
    t = MEASURED[n]
    near = [max(k for k in t if k <= chunks), min(k for k in t if k >= chunks)]
    assert max(t[k] for k in near) <= 1.15 * min(t.values())


@pytest.mark.parametrize("cols,nz,slots", [(1, 4, 608), (1, 2, 608), (1, 500, 608), (4000, 3, 912),
                                           (100000, 64, 912)])
def test_chunks_stay_in_range(march_zc, cols, nz, slots):
    assert 2 <= march_zc(cols, nz, slots, 6) <= max(2, min(56, nz))

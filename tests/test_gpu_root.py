"""The J2 law's root and inverse root (rf_law.cuh, root_pair) against FP64 square roots.

Bounds, relative, in units of u = 2^-24 (half a unit in the last place of 1). The hardware's
reciprocal root is good to 2^-22.4 at worst; Goldschmidt's step squares that away and leaves the
roundings of its operations: g = x r one, e = 1/2 - g h one more that counts twice (it carries
g's), so h ends within 3 u. The root is corrected by its residual (exact in one fused operation),
which leaves the last rounding and half of what the inverse is off of a correction of 2 u: 1.5 u. Of
subnormal x the residual itself is rounded to multiples of 2^-149, which can leave the uncorrected
root's 3 u.
"""

import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "rf_law.cuh"
__global__ void k(const float* x, float* r, float* i, int n) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x)
    rfk::root_pair(x[t], r[t], i[t]);
}
extern "C" int run(const float* x, float* r, float* i, int n) {
  k<<<304, 256>>>(x, r, i, n);
  return (int)cudaDeviceSynchronize();
}
"""

U = 2.0 ** -24


@pytest.fixture(scope="module")
def roots(tmp_path_factory):
    import torch
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("root")
    (d / "root.cu").write_text(SRC)
    from paper_2103_10203_gb300.build import ARCH, CSRC, NVCC_FLAGS
    subprocess.run([nvcc, *ARCH, *NVCC_FLAGS, "-shared", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), str(d / "root.cu"), "-o", str(d / "root.so")],
                   check=True)
    lib = C.CDLL(str(d / "root.so"))

    def run(x):
        x = torch.as_tensor(np.ascontiguousarray(x, np.float32), device="cuda")
        r, i = torch.empty_like(x), torch.empty_like(x)
        torch.cuda.synchronize()
        assert lib.run(*[C.c_void_p(t.data_ptr()) for t in (x, r, i)], x.numel()) == 0
        return r.cpu().numpy().astype(np.float64), i.cpu().numpy().astype(np.float64)

    return run


def floats(lo, hi, n, seed):
    """n positive floats spread over the bit patterns lo..hi, the ends among them."""
    b = np.random.default_rng(seed).integers(lo, hi, n, dtype=np.int64)
    b[:2] = lo, hi - 1
    return b.astype(np.uint32).view(np.float32)


def test_normal_numbers(roots):
    x = floats(0x00800000, 0x7f800000, 1 << 22, 1)
    r, i = roots(x)
    want = np.sqrt(x.astype(np.float64))
    assert np.abs(r / want - 1.0).max() <= 1.5 * U
    assert np.abs(i * want - 1.0).max() <= 3.0 * U


def test_subnormal_numbers(roots):
    x = floats(1, 0x00800000, 1 << 20, 2)
    r, i = roots(x)
    want = np.sqrt(x.astype(np.float64))
    assert np.abs(r / want - 1.0).max() <= 3.0 * U
    assert np.abs(i * want - 1.0).max() <= 3.0 * U


def test_zero_and_infinity(roots):
    r, i = roots(np.array([0.0, np.inf], np.float32))
    assert r[0] == 0.0 and np.isfinite(i[0])
    assert np.isnan(r[1])   # a yielding phase hands this on to its stress

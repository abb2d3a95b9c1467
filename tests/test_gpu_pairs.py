"""The float pairs that FP64 fields become (ff_of_double) and their way back: a small
kernel over the library's own header.  hi is the nearest float and lo the nearest float
of the rest, so with 2^E <= |v| < 2^(E+1) the pair is within 2^-25 2^-24 2^(E+1) of v;
scaling by 2^k is exact either way."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1405_6456_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = r"""
#include "kernels.cuh"
__global__ void pairs(int n, const double* v, int k, float2* p, double* back) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  p[i] = ofd::ff_of_double(v[i], k);
  back[i] = ofd::double_of_float(p[i].x, k) + ofd::double_of_float(p[i].y, k);
}
extern "C" int run(int n, const void* v, int k, void* p, void* back) {
  pairs<<<(n + 255) / 256, 256>>>(n, (const double*)v, k, (float2*)p, (double*)back);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("pairs")
    src, so = os.path.join(d, "pairs.cu"), os.path.join(d, "pairs.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([B._nvcc(), *B.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared", "-Xcompiler",
                    "-fPIC", "-I", B.CSRC, "-o", so, src], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("k", [0, 40, -300, 511])
def test_pairs_are_nearest_and_scale_exactly(lib, k):
    rng = np.random.default_rng(1)
    n = 1 << 18
    w = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-69, 120, n)) * rng.choice([-1.0, 1.0], n)
    # a carry through the mantissa into the exponent, ties, exact floats, the range's ends
    w[:12] = [2.0 - 2.0**-52, 1.0 + 2.0**-24, 1.0 - 2.0**-25, -1.0 - 3 * 2.0**-24, 1.0, 2.0**-70, 0.0, -0.0,
              2.0**127 - 2.0**74, 2.0**-70 + 2.0**-122, 1.0 + 2.0**-52, -(2.0 - 2.0**-25)]
    v = torch.as_tensor(np.ldexp(w, k), device="cuda:0")
    p = torch.empty((n, 2), dtype=torch.float32, device="cuda:0")
    back = torch.empty(n, dtype=torch.float64, device="cuda:0")
    assert lib.run(n, ctypes.c_void_p(v.data_ptr()), k, ctypes.c_void_p(p.data_ptr()),
                   ctypes.c_void_p(back.data_ptr())) == 0
    p = p.cpu().numpy().astype(np.float64)
    near = w.astype(np.float32).astype(np.float64)
    assert np.array_equal(np.abs(w - p[:, 0]), np.abs(w - near))  # (equal at ties)
    top = np.ldexp(1.0, np.frexp(w)[1])
    assert (np.abs(w - p.sum(1)) <= 2.0**-49 * top).all()
    assert np.array_equal(back.cpu().numpy(), np.ldexp(p.sum(1), k))

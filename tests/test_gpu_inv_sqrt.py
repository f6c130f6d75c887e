"""The reciprocal square root of the LP_FP64 factor (inv_sqrt): an approximation
and one step of Halley's iteration.

Error bound: e = 1 - v y^2 is off by 2^-53 (the product v y; the multiply-add
rounds far below), which enters the result halved, 2^-54; the step leaves
5/16 e^3 < 2^-55 for an approximation good to 18 bits, and rounds once, 2^-53.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SOURCE = r"""
#include "lp_internal.cuh"
__global__ void k_both(long n, const double* v, double* own, double* ref) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += gridDim.x * (long)blockDim.x) {
    own[i] = lp::inv_sqrt(v[i]);
    ref[i] = rsqrt(v[i]);
  }
}
extern "C" int both(long n, const double* v, double* own, double* ref) {
  k_both<<<608, 256>>>(n, v, own, ref);
  return (int)cudaDeviceSynchronize();
}
"""


def test_inv_sqrt_over_the_normal_numbers(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_14061_gb300 import build
    src, out = tmp_path / "inv_sqrt.cu", str(tmp_path / "inv_sqrt.so")
    src.write_text(SOURCE)
    subprocess.run([build.NVCC] + build.FLAGS + ["-I" + build.SRC, "-shared", "-cudart", "shared",
                                                 "-o", out, str(src)], check=True)
    f = ctypes.CDLL(out).both
    f.argtypes = [ctypes.c_long] + [ctypes.c_void_p] * 3
    rng = np.random.default_rng(1)
    m = rng.integers(0, 2 ** 52, 4_000_000, dtype=np.uint64)
    e = rng.integers(1, 2047, m.size, dtype=np.uint64)
    edge = np.array([0, 1, 2, 2 ** 51, 2 ** 52 - 2, 2 ** 52 - 1], dtype=np.uint64)  # every exponent
    m = np.concatenate([m, np.tile(edge, 2046)])
    e = np.concatenate([e, np.repeat(np.arange(1, 2047, dtype=np.uint64), edge.size)])
    v = (m | (e << np.uint64(52))).view(np.float64)
    d = torch.tensor(v, device="cuda:0")
    own, ref = torch.empty_like(d), torch.empty_like(d)
    torch.cuda.synchronize()
    assert f(d.numel(), d.data_ptr(), own.data_ptr(), ref.data_ptr()) == 0
    L = np.longdouble
    exact = 1 / np.sqrt(v.astype(L))
    unit = exact * L(2) ** -53
    err = [float(np.abs((t.cpu().numpy().astype(L) - exact) / unit).max()) for t in (own, ref)]
    print(f"largest errors in 2^-53: inv_sqrt {err[0]:.3f}, rsqrt {err[1]:.3f}")
    assert err[0] <= 1.0 + 0.5 + 0.25

"""The FP64 building blocks of csrc/dg_math64.cuh against CUDA's own functions.

One third-order step on a hardware approximation of relative error d leaves at most about d^3; the
approximations carry 20 bits, so the result is CUDA's correctly rounded one to within the roundings
of the last operations: one unit in the last place for the reciprocal, two for the square roots.
Zeros, infinities, NaNs, subnormals and extreme exponents must give CUDA's results exactly, and the
bit-pattern comparisons must agree with the floating-point ones, NaNs included."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "dg_math64.cuh"
using namespace dgpf;
__global__ void k(const double *x, const double *y, double *o, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const double a = x[t], b = y[t], A = fabs(a), B = fabs(b);
  double *r = o + 20 * (long)t;
  r[0] = rcp64(a);            r[1] = 1.0 / a;
  r[2] = rsqrt64(A);          r[3] = rsqrt(A);
  r[4] = sqrt64(A);           r[5] = sqrt(A);
  r[6] = max_nonneg64(A, B);  r[7] = fmax(A, B);
  r[8] = nonpositive64(a);    r[9] = a <= 0.0;
  r[10] = finite64(a);        r[11] = isfinite(a);
  r[12] = has_gradient(A);    r[13] = A >= 1e-24;
  r[14] = rcp64_rn(a);        r[15] = 1.0 / a;
  r[16] = div64_rn(b, a, rcp64_rn(a));  r[17] = b / a;
  r[18] = sqrt64_rn(A);       r[19] = sqrt(A);
}
extern "C" int run(const double *x, const double *y, double *o, int n) {
  k<<<(n + 255) / 256, 256>>>(x, y, o, n);
  return (int)cudaDeviceSynchronize();
}
"""


def test_math64(tmp_path):
    import torch
    from paper_2306_05002_gb300 import build
    src, lib = tmp_path / "m.cu", tmp_path / "m.so"
    src.write_text(SRC)
    subprocess.run([build.nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I" + build.CSRC,
                                                  str(src), "-o", str(lib)], check=True)
    rng = np.random.default_rng(0)
    x = rng.uniform(1.0, 2.0, 1 << 20) * 2.0 ** rng.integers(-60, 60, 1 << 20) * rng.choice([-1.0, 1.0], 1 << 20)
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 1e-310, 2.2250738585072014e-308, 1e-300,
                        1e300, -1e300, 1.7e308, 1e-24, np.nextafter(1e-24, 0), np.nextafter(1e-24, 1), 1.0, 2.0 ** 500,
                        2.0 ** 501, 2.0 ** -500, 2.0 ** -501, np.nextafter(1.0, 0), np.nextafter(1.0, 2), np.nextafter(1024.0, 0),
                        np.nextafter(-1.0, 0)])
    sx, sy = [g.ravel() for g in np.meshgrid(special, special)]
    x = np.concatenate([x, sx])
    y = np.concatenate([rng.permutation(x[:1 << 20]), sy])
    dx, dy = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    out = torch.zeros((len(x), 20), dtype=torch.float64, device="cuda")
    fn = ctypes.CDLL(str(lib)).run
    fn.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    assert fn(dx.data_ptr(), dy.data_ptr(), out.data_ptr(), len(x)) == 0
    r = out.cpu().numpy()
    for c, ulp in ((0, 1), (2, 2), (4, 2)):
        got, ref = r[: 1 << 20, c], r[: 1 << 20, c + 1]
        assert np.max(np.abs(got - ref) / np.spacing(np.abs(ref))) <= ulp, c
        plain = np.isin(np.abs(x), (1.0, np.nextafter(1.0, 0), np.nextafter(1.0, 2), np.nextafter(1024.0, 0), 2.0 ** 500, 2.0 ** -500, 1e-24)) | (np.abs(x) < 1.1e-24) & (np.abs(x) > 0.9e-24)
        far = ~plain
        far[: 1 << 20] = False
        assert np.array_equal(r[far, c], r[far, c + 1], equal_nan=True), c
    for c in (14, 16, 18):  # the correctly rounded forms: CUDA's bits (a quotient's sign of zero aside)
        got, ref = r[:, c], r[:, c + 1]
        bad = ~((got == ref) | (np.isnan(got) & np.isnan(ref)))
        assert not bad.any(), (c, bad.sum(), x[bad][:5], y[bad][:5], got[bad][:5], ref[bad][:5])
    for c in (6, 8, 10, 12):
        assert np.array_equal(r[:, c], r[:, c + 1], equal_nan=True), c

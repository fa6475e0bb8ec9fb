"""The correctly rounded forms of csrc/dg_math64.cuh (sqrt64_rn, rcp64_rn, div64_rn) against CUDA's own
functions, bit for bit: on 2^30 random arguments, compared on the device, and on square roots that lie
next to a rounding boundary.

The hard arguments: with S a 53-bit integer and j a small even one, x = S^2 + S + j has its root within
(|j| + 1/4) / (2 S) of S + 1/2, the boundary between S and S + 1.  x is a 53-bit number times 2^52 or
2^53 exactly when S^2 + S + j = 0 modulo that power, which Newton's iteration on the 2-adic integers
solves.  A root whose last correction carries a relative error of 2^-20 is rounded the wrong way on
most of them."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "dg_math64.cuh"
using namespace dgpf;
__device__ unsigned long long mix(unsigned long long z) {  // splitmix64
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
// significand bits of r, exponent -60 .. 67
__device__ double number(unsigned long long r) {
  return __longlong_as_double((long long)((r & 0xfffffffffffffull) | (963ull + (r >> 57)) << 52));
}
__device__ void check(double a, double b, unsigned long long *bad) {
  if (sqrt64_rn(a) != sqrt(a)) atomicAdd(bad, 1ull);
  if (rcp64_rn(a) != 1.0 / a) atomicAdd(bad + 1, 1ull);
  if (div64_rn(b, a, rcp64_rn(a)) != b / a) atomicAdd(bad + 2, 1ull);
}
__global__ void k_random(unsigned long long seed, int n, unsigned long long *bad) {
  for (int k = 0; k < n; ++k) {
    const unsigned long long t = seed + ((unsigned long long)k * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x;
    check(number(mix(2 * t)), number(mix(2 * t + 1)), bad);
  }
}
__global__ void k_given(const double *x, int n, unsigned long long *bad) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) check(x[t], x[n - 1 - t], bad);
}
extern "C" int run_random(unsigned long long seed, int blocks, int n, unsigned long long *bad) {
  k_random<<<blocks, 256>>>(seed, n, bad);
  return (int)cudaDeviceSynchronize();
}
extern "C" int run_given(const double *x, int n, unsigned long long *bad) {
  k_given<<<(n + 255) / 256, 256>>>(x, n, bad);
  return (int)cudaDeviceSynchronize();
}
"""


def hard_roots(seed=0, per=60000):
    rng = np.random.default_rng(seed)
    out = []
    for K in (52, 53):
        bits = rng.integers(1, 30, per)
        js = 2 * (1 + (rng.integers(0, 2 ** 30, per) >> bits)) * rng.choice([-1, 1], per)
        for r0 in (0, 1):
            # S <- S - f(S) / f'(S) modulo 2^64, f = S^2 + S + j, f' = 2 S + 1 odd
            S = np.full(per, r0, np.uint64)
            j = js.astype(np.int64).view(np.uint64)
            for _ in range(7):
                fp = 2 * S + np.uint64(1)
                inv = fp.copy()
                for _ in range(6):
                    inv = inv * (np.uint64(2) - fp * inv)
                S = S - (S * S + S + j) * inv
            S &= np.uint64(2 ** K - 1)
            for s, jj in zip(S.tolist(), js.tolist()):
                s |= 2 ** 52  # (K = 52: the significand's leading bit is free)
                x = s * s + s + jj
                if K == 52 and x % 2 ** 52 == 0 or K == 53 and x % 2 ** 53 == 0:
                    m = x >> K
                    if 2 ** 52 <= m < 2 ** 53:
                        out.append(float(m) * 2.0 ** (K - 52))
    return np.array(out)


def test_correctly_rounded(tmp_path):
    import torch
    from paper_2306_05002_gb300 import build
    x = hard_roots()
    assert len(x) > 40000
    ones = (2.0 ** 53 - 1 - np.arange(4)) * 2.0 ** np.arange(-80, 80)[:, None]  # significands of (almost) all ones
    first = (2.0 ** 52 + np.arange(4)) * 2.0 ** np.arange(-80, 80)[:, None]  # 1, 1 + 2^-52, ...
    x = np.concatenate([x, x * 2.0 ** -40, x * 2.0 ** 60, ones.ravel(), first.ravel()])
    src, lib = tmp_path / "m.cu", tmp_path / "m.so"
    src.write_text(SRC)
    subprocess.run([build.nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I" + build.CSRC,
                                                  str(src), "-o", str(lib)], check=True)
    so = ctypes.CDLL(str(lib))
    bad = torch.zeros(3, dtype=torch.int64, device="cuda")
    d = torch.from_numpy(x).cuda()
    assert so.run_given(ctypes.c_void_p(d.data_ptr()), len(x), ctypes.c_void_p(bad.data_ptr())) == 0
    assert bad.tolist() == [0, 0, 0], f"of {len(x)} arguments: {bad.tolist()} roots, reciprocals, quotients"
    # 1024 blocks of 256 threads, 4096 arguments each
    assert so.run_random(ctypes.c_ulonglong(12345), 1024, 4096, ctypes.c_void_p(bad.data_ptr())) == 0
    assert bad.tolist() == [0, 0, 0], f"of 2^30 arguments: {bad.tolist()} roots, reciprocals, quotients"

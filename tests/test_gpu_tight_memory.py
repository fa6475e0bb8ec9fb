"""Workspaces where device memory does not hold the larger form of them: the call falls back on the smaller
form and gives the same results.

The failure is made on the host: the library's objects are linked a second time with cudaMalloc wrapped by a
function that refuses one given size, and a child process runs on that copy."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2306_05002_gb300 import workloads as W
from tests.helpers import problem
from tests.test_gpu_fp32bulk import TOL32, _l2, _storage_bound

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WRAP = r"""
#include <cuda_runtime_api.h>
extern "C" cudaError_t __real_cudaMalloc(void **p, size_t n);
static size_t refused = 0;
static int times = 0;
extern "C" void refuse(size_t n) { refused = n; times = 0; }
extern "C" int refusals() { return times; }
extern "C" cudaError_t __wrap_cudaMalloc(void **p, size_t n) {
  if (n == refused) {
    ++times;
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  return __real_cudaMalloc(p, n);
}
"""
CHILD = r"""
import ctypes, sys
import numpy as np, torch
import paper_2306_05002_gb300 as dg
from paper_2306_05002_gb300 import workloads as W
lib = dg.load(sys.argv[1])
lib.refuse.argtypes = [ctypes.c_size_t]
size, out = int(sys.argv[2]), {}
def run(tag, expect):
    lib.refuse(size if expect else 0)
    exec(BODY, dict(dg=dg, W=W, torch=torch, tag=tag, out=out))
    assert (lib.refusals() > 0) == expect, (tag, lib.refusals())
BODY = open(sys.argv[3]).read()
run("plain", False)
run("tight", True)
np.savez(sys.argv[4], **out)
"""


@pytest.fixture(scope="module")
def wrapped(tmp_path_factory):
    from paper_2306_05002_gb300 import build
    build.build()
    d = tmp_path_factory.mktemp("wrapped")
    src, lib = d / "wrap.cu", d / "libwrapped.so"
    src.write_text(WRAP)
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    subprocess.run([build.nvcc()] + build.ARCH + ["-shared", "-Xcompiler", "-fPIC", "-Xlinker", "--wrap=cudaMalloc",
                                                  str(src)] + objs + ["-o", str(lib)], check=True)
    return str(lib)


def _both(wrapped, tmp_path, size, body):
    """Results of `body` with every allocation granted, and with those of `size` bytes refused."""
    (tmp_path / "body.py").write_text(body)
    r = subprocess.run([sys.executable, "-c", CHILD, wrapped, str(size), str(tmp_path / "body.py"),
                        str(tmp_path / "out.npz")], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    return np.load(tmp_path / "out.npz")


@pytest.mark.parametrize("p", [1, 3, 5])
def test_kinematic_mode_with_one_trace_buffer(dg, wrapped, tmp_path, p):
    """A volume and a stage launch per stage instead of the fused one: the same operations on the same
    operands."""
    n = 37
    size = 2 * 3 * n * n * 4 * (p + 1) * 8  # two buffers of three fields per face node
    r = _both(wrapped, tmp_path, size, f"""
wl = W.rider_kothe(n={n}, p={p})
s = dg.KinematicSolver(wl)
w = torch.from_numpy(wl.w.copy()).cuda()
out[tag + "_rhs"] = s.dg_kin_rhs(w, 0.3).cpu().numpy()
for k in (1, 8, 11):
    s.dg_kin_step(w, 0.1 * k, wl.dt, k)
    out[tag + "_%d" % k] = w.cpu().numpy()
assert s.dg_status_read() == 0
s.close()
""")
    for k in ("rhs", "1", "8", "11"):
        assert np.array_equal(r["plain_" + k], r["tight_" + k]), k


@pytest.mark.parametrize("dim,p", [(1, 3), (2, 1), (2, 4)])
def test_reinitialisation_with_one_trace_buffer(dg, wrapped, tmp_path, dim, p):
    n = 37 if dim == 2 else 301
    nfk = 4 * n * n * (p + 1) if dim == 2 else 2 * n
    size = 2 * 2 * nfk * 8  # two buffers of two fields per face node
    make = f"W.drop_2d({n}, {p})" if dim == 2 else f"W.slab_1d({n}, {p})"
    r = _both(wrapped, tmp_path, size, f"""
wl = {make}
s = dg.Solver(wl)
w = torch.from_numpy(wl.w.copy()).cuda()
for k in (1, 4):
    s.dg_reinit(w, k)
    out[tag + "_%d" % k] = w.cpu().numpy()
s.close()
""")
    for k in ("1", "4"):
        assert np.array_equal(r["plain_" + k], r["tight_" + k]), k


def test_fp32bulk_without_room_for_the_line_kernels(orc, dg, wrapped, tmp_path):
    """p = 5: the tiles' face records take more than the one-node kernels'.  The right-hand side is held
    to the oracle as that of any FP32-bulk context, eight steps to the mode's accuracy target against the
    context with line kernels."""
    n, p = 71, 5
    size = (n * n + 4) // 5 * 4 * 3 * 32 * 4 * 4  # floats of the tiles' face records, in bytes
    assert size > 12 * 4 * (p + 1) * n * n * 4
    r = _both(wrapped, tmp_path, size, f"""
wl = W.drop_2d({n}, {p})
s = dg.Solver(wl, precision="fp32bulk")
out[tag + "_lines"] = s.dg_line_kernels(8)
w = torch.from_numpy(wl.w.copy()).cuda()
out[tag + "_rhs"] = s.dg_rhs(w).cpu().numpy()
s.dg_step(w, wl.dt, 8)
out[tag + "_w"] = w.cpu().numpy()
assert s.dg_status_read() == 0
s.close()
""")
    assert (r["plain_lines"], r["tight_lines"]) == (1, 0)
    wl = W.drop_2d(n, p)
    pb = problem(orc, wl)
    L_ref, S = orc.rhs(pb, wl.w, want_scale=True)
    extra = _storage_bound(orc, wl, wl.w)
    for v in range(7):
        assert np.abs(r["tight_rhs"][v] - L_ref[v]).max() <= TOL32 * S[v].max() + extra.get(v, 0.0), v
    assert _l2(r["tight_w"][0], r["plain_w"][0]) <= 1e-5
    assert _l2(orc.primitives(pb, r["tight_w"])[3], orc.primitives(pb, r["plain_w"])[3]) <= 1e-5

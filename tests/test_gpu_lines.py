"""The FP32-bulk kernels with one element line per thread (csrc/dg_lines32.cuh), which single problems
run from a few line warps per SM on: one right-hand side against the FP64 oracle on meshes just above
that limit, of odd and unequal sides (ragged last tile), for every order, with walls of every kind,
gravity, viscous stress and surface tension; steps against the FP64 path; failure flags.

Tolerances: those of the one-node-per-thread kernels (tests/test_gpu_fp32bulk.py), which hold for any
order of the FP32 operations where the level set is continuous across the faces (so the bubble's
column is closed by walls in y: across a periodic pair there both kernels carry the FP32 error of
lambda through its jump, 1.8e-5 of the scale at p = 2)."""
import numpy as np
import pytest

from paper_2306_05002_gb300 import workloads as W
from tests.helpers import problem
from tests.test_gpu_fp32bulk import _l2, _rhs32, _run

pytestmark = pytest.mark.gpu
# (nx, ny) with 3/2 (p = 1), 4 (p = 2) or 5 line warps for each of 152 SMs
MESH = {1: (57, 65), 2: (71, 87), 3: (71, 87), 4: (61, 77), 5: (59, 65)}


def _bubble(p, terms, bc):
    nx, ny = MESH[p]
    wl = W.rising_bubble(nx=nx, ny=ny, p=p, nquad=60)
    wl.viscous, wl.surface_tension = "viscous" in terms, "tension" in terms
    wl.bc = bc
    wl.p_bc = tuple(1e5 if b == "pressure" else 0.0 for b in bc)
    x, y = W.node_coords(wl)
    u, v = 0.3 * np.sin(2 * np.pi * x) * np.cos(np.pi * y), 0.2 * np.cos(2 * np.pi * x) * np.sin(np.pi * y)
    rho = wl.w[2] + wl.w[3]
    w = wl.w.copy()
    w[4], w[5] = rho * u, rho * v
    w[6] += 0.5 * rho * (u * u + v * v)
    wl.w = w
    return wl


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("terms,bc", [((), ("noslip", "slip", "pressure", "noslip")),
                                      (("viscous",), ("slip", "slip", "noslip", "pressure")),
                                      (("tension",), ("periodic", "periodic", "slip", "noslip")),
                                      (("viscous", "tension"), ("pressure", "noslip", "noslip", "slip"))])
def test_rhs_lines(orc, dg, p, terms, bc):
    _rhs32(orc, dg, _bubble(p, terms, bc))


@pytest.mark.parametrize("p,n", [(1, 61), (2, 79), (3, 79), (4, 69), (5, 62)])
@pytest.mark.parametrize("steps", [1, 3])
def test_steps_lines_track_fp64(orc, dg, p, n, steps):
    """A single step (FP64 in and out) and a call of several (float-float step start carried)."""
    wl = W.drop_2d(n=n, p=p, seed=3, water_inside=p % 2 == 0)
    w64, w32 = _run(dg, wl, "fp64", steps), _run(dg, wl, "fp32bulk", steps)
    pb = problem(orc, wl)
    assert _l2(w32[0], w64[0]) <= 1e-6
    assert _l2(orc.primitives(pb, w32)[3], orc.primitives(pb, w64)[3]) <= 1e-6


def test_lines_flag_failures(dg):
    import torch
    wl = W.drop_2d(n=80, p=3, seed=2)
    s = dg.Solver(wl, precision="fp32bulk")
    for field, value, code in ((0, np.nan, -5), (3, -1e4, -6)):
        w = wl.w.copy()
        w[field, wl.N - 1] = value  # the last node, in the ragged tile
        d = torch.from_numpy(w).cuda()
        s.dg_step(d, wl.dt, 1)
        assert s.dg_status_read() == code
    d = torch.from_numpy(wl.w.copy()).cuda()
    s.dg_step(d, wl.dt, 2)
    assert s.dg_status_read() == 0
    s.close()

"""Which calls run the FP32-bulk line kernels (use_lines32, csrc/dg_lines32.cuh), and that they and the
one-node-per-thread kernels serve the calls of one context side by side.

Mesh sizes are given in line warps per SM of the GPU at hand; the element counts leave a ragged last tile
and an odd number of tiles, so that the last block's second warp has none.  The routes held here are those
whose other choice measured 6 to 60% slower.  Tolerances: the right-hand side as the one-node kernels'
(tests/test_gpu_fp32bulk.py), steps within 1e-5 (relative L2) of the FP64 path in phi and P, the mode's
accuracy target."""
import numpy as np
import pytest

from paper_2306_05002_gb300 import workloads as W
from tests.helpers import problem
from tests.test_gpu_fp32bulk import TOL32, _l2, _rhs32, _storage_bound

pytestmark = pytest.mark.gpu
TERMS = {"none": (False, False), "tension": (False, True), "viscous": (True, False), "both": (True, True)}


def _side(p, warps):
    """n of an n x n mesh of about `warps` line warps per SM: a ragged last tile, an odd number of tiles."""
    import torch
    sms, per = torch.cuda.get_device_properties(0).multi_processor_count, 32 // (p + 1)
    n = int(round((warps * sms * per) ** 0.5))
    return next(m for m in range(n, n + 40) if m * m % per and m * m // per % 2 == 0)


def _mesh(p, warps, terms):
    n = _side(p, warps)
    v, t = TERMS[terms]
    return W.Workload(name="mesh", dim=2, nx=n, ny=n, p=p, viscous=v, surface_tension=t, mu=(1e-2, 1e-1), sigma=0.07)


def _flow(p, warps, terms):
    """A periodic drop, or, with viscous stress, a Rayleigh-Taylor column between walls."""
    n = _side(p, warps)
    v, t = TERMS[terms]
    wl = W.rayleigh_taylor(n=n, p=p, seed=3) if v else W.drop_2d(n=n, p=p, seed=2)
    wl.viscous, wl.surface_tension = v, t
    if t and not v:
        wl.sigma = 0.07
    return wl


def _bubble(p, warps, terms):
    """A moving bubble in a column closed by walls in y (tests/test_gpu_lines.py)."""
    n = _side(p, warps)
    wl = W.rising_bubble(nx=n, ny=n, p=p, nquad=60)
    wl.viscous, wl.surface_tension = TERMS[terms]
    wl.bc = ("periodic", "periodic", "slip", "noslip")
    x, y = W.node_coords(wl)
    u, v = 0.3 * np.sin(2 * np.pi * x) * np.cos(np.pi * y), 0.2 * np.cos(2 * np.pi * x) * np.sin(np.pi * y)
    rho = wl.w[2] + wl.w[3]
    w = wl.w.copy()
    w[4], w[5] = rho * u, rho * v
    w[6] += 0.5 * rho * (u * u + v * v)
    wl.w = w
    return wl


def _routes(dg, wl):
    s = dg.Solver(wl, precision="fp32bulk")
    r = [s.dg_line_kernels(k) for k in (0, 1, 2, 8, 20)]
    s.close()
    return r


# p, terms, line warps per SM: (dg_rhs, 1 step, 2 steps, 8 steps)
@pytest.mark.parametrize("p,terms,warps,want", [
    (1, "none", 1.0, (0, 0, 0, 0)), (1, "none", 2.2, (0, 0, 0, 1)), (1, "none", 5.2, (1, 1, 1, 1)),
    (1, "both", 1.8, (0, 1, 1, 1)),
    (2, "none", 5.2, (1, 0, 0, 0)), (2, "tension", 3.0, (1, 0, 0, 0)), (2, "none", 7.0, (1, 1, 1, 1)),
    (2, "viscous", 1.8, (0, 0, 0, 1)), (2, "both", 5.2, (1, 1, 1, 1)),
    (3, "none", 4.5, (0, 0, 0, 0)), (3, "none", 8.0, (1, 1, 1, 1)), (3, "both", 6.5, (1, 0, 0, 0)),
    (3, "viscous", 9.0, (1, 1, 1, 1)), (3, "none", 13.2, (0, 0, 0, 0)), (3, "none", 30.0, (0, 0, 1, 1)),
    (3, "both", 30.0, (0, 0, 0, 1)),
    (4, "none", 5.4, (1, 0, 0, 0)), (4, "none", 10.0, (1, 1, 1, 1)), (4, "both", 10.0, (0, 1, 1, 1)),
    (4, "tension", 10.0, (1, 1, 1, 1)),
    (4, "none", 27.0, (0, 0, 1, 1)), (4, "both", 27.0, (0, 0, 0, 1)),
    (5, "none", 5.1, (0, 0, 0, 0)), (5, "none", 6.6, (1, 0, 0, 1)), (5, "both", 6.6, (1, 1, 1, 1)),
    (5, "none", 27.0, (0, 0, 0, 1)), (5, "both", 27.0, (0, 0, 0, 0))])
def test_routes(dg, p, terms, warps, want):
    assert tuple(_routes(dg, _mesh(p, warps, terms))) == want + want[3:]


def test_line_kernels_query(dg):
    from paper_2306_05002_gb300 import load
    assert load().dg_line_kernels(None, 1) == -1
    s = dg.Solver(_mesh(1, 5.2, "none"))
    assert [s.dg_line_kernels(k) for k in (0, 1, 8)] == [0, 0, 0]
    with pytest.raises(dg.DGError):
        s.dg_line_kernels(-1)
    s.close()
    s = dg.Solver(W.slab_1d(nx=4000, p=3), precision="fp32bulk")
    assert [s.dg_line_kernels(k) for k in (0, 8)] == [0, 0]
    s.close()


# one wave of line warps, and several (launched plainly, with non-coherent loads)
@pytest.mark.parametrize("p,terms,warps", [(1, "none", 5.2), (1, "both", 26.2), (2, "tension", 7.0), (2, "none", 26.2),
                                           (2, "both", 26.2), (3, "none", 6.0), (3, "both", 6.0), (4, "viscous", 5.4),
                                           (4, "none", 6.0), (5, "none", 6.4), (5, "both", 6.4)])
def test_rhs_on_lines(orc, dg, p, terms, warps):
    wl = _bubble(p, warps, terms)
    assert _routes(dg, wl)[0] == 1
    _rhs32(orc, dg, wl)


@pytest.mark.parametrize("p,terms,warps", [(1, "none", 2.2), (1, "none", 26.2), (1, "both", 26.2), (2, "viscous", 2.3),
                                           (2, "none", 26.2), (2, "both", 26.2), (3, "none", 26.2), (3, "tension", 26.2),
                                           (3, "both", 26.2), (4, "none", 26.2), (4, "viscous", 26.2),
                                           (4, "both", 26.2), (5, "none", 6.6), (5, "none", 26.2)])
def test_steps_by_length_track_fp64(orc, dg, p, terms, warps):
    """Calls of 8, 1, 9 and 2 steps on one context (sequences of eight on lines, the single and the
    remainder on either), then a right-hand side, against the FP64 path."""
    import torch
    wl = _flow(p, warps, terms)
    assert _routes(dg, wl)[3] == 1
    s64, s32 = dg.Solver(wl), dg.Solver(wl, precision="fp32bulk")
    a, b = torch.from_numpy(wl.w.copy()).cuda(), torch.from_numpy(wl.w.copy()).cuda()
    pb = problem(orc, wl)
    for n in (8, 1, 9, 2):
        s64.dg_step(a, wl.dt, n)
        s32.dg_step(b, wl.dt, n)
        wa, wb = a.cpu().numpy(), b.cpu().numpy()
        assert _l2(wb[0], wa[0]) <= 1e-5
        assert _l2(orc.primitives(pb, wb)[3], orc.primitives(pb, wa)[3]) <= 1e-5
    assert s32.dg_status_read() == 0
    L = s32.dg_rhs(b)
    fresh = dg.Solver(wl, precision="fp32bulk")  # nothing of the calls before is left in the arrays
    assert torch.equal(L, fresh.dg_rhs(b))
    for s in (s64, s32, fresh):
        s.close()


@pytest.mark.parametrize("p,warps", [(1, 2.2), (2, 7.0), (3, 8.0), (3, 26.2), (4, 10.0), (5, 6.6)])
def test_failures_in_the_ragged_tile(dg, p, warps):
    """A NaN and a negative density at the last node of the mesh, in the partial tile, seen by a sequence
    on lines; a sound state after it leaves the status clear (the tile's padding slots hold no failure)."""
    import torch
    wl = _flow(p, warps, "none")
    assert wl.E % (32 // (p + 1)) != 0
    s = dg.Solver(wl, precision="fp32bulk")
    assert s.dg_line_kernels(8) == 1
    for field, value, code in ((0, np.nan, -5), (3, -1e4, -6)):
        w = wl.w.copy()
        w[field, wl.N - 1] = value
        s.dg_step(torch.from_numpy(w).cuda(), wl.dt, 8)
        assert s.dg_status_read() == code
    s.dg_step(torch.from_numpy(wl.w.copy()).cuda(), wl.dt, 8)
    assert s.dg_status_read() == 0
    s.close()


@pytest.mark.parametrize("p,warps", [(1, 5.2), (2, 7.0), (3, 9.0), (4, 6.0), (5, 6.6)])
@pytest.mark.parametrize("phase", [0, 1])
def test_viscosity_of_a_pure_phase(orc, dg, p, warps, phase):
    """One phase alone, of 1e-8 times the other's viscosity: the mixture's is its own.  The rows that
    viscosity enters, momentum and energy (those of the absent phase are zero to the oracle's rounding)."""
    import torch
    n = _side(p, warps)
    wl = W.Workload(name="pure", dim=2, nx=n, ny=n, p=p, viscous=True, mu=(1e5, 1e13) if phase == 0 else (1e13, 1e5))
    x, y = W.node_coords(wl)
    wl.w = W.conserved(wl, np.full(wl.N, 1.0 - phase), 0.2 * np.sin(2 * np.pi * y), 1e5,
                       0.3 * np.sin(2 * np.pi * y), 0.2 * np.cos(2 * np.pi * x))
    assert _routes(dg, wl)[0] == 1
    L_ref, S = orc.rhs(problem(orc, wl), wl.w, want_scale=True)
    s = dg.Solver(wl, precision="fp32bulk")
    L = s.dg_rhs(torch.from_numpy(wl.w.copy()).cuda()).cpu().numpy()
    s.close()
    extra = _storage_bound(orc, wl, wl.w)
    for v in (4, 5, 6):
        assert np.abs(L[v] - L_ref[v]).max() <= TOL32 * S[v].max() + extra.get(v, 0.0), v

"""Kinematic mode on a state with a NaN level-set value: where the right-hand side is NaN and where it
is not.

On triangles n = grad psi / |grad psi| is taken as zero where |grad psi| < 1e-12, which a NaN is not, so
the NaN reaches the phase field through the normals of the triangle and of its neighbours' edges, as in
the oracle.  On rectangles n is zero unless |grad psi| >= 1e-12: the phase field's right-hand side stays
what the finite part of the state gives.  Either way psi itself is NaN and the status word says so."""
import numpy as np
import pytest

from paper_2306_05002_gb300 import workloads as W
from tests.test_gpu_triangles import _kin

pytestmark = pytest.mark.gpu


def _rhs(dg, wl, w):
    import torch
    s = dg.KinematicSolver(wl)
    L = s.dg_kin_rhs(torch.from_numpy(w).cuda(), 0.7).cpu().numpy()
    d = torch.from_numpy(w).cuda()
    s.dg_kin_step(d, 0.0, wl.dt, 1)
    status = s.dg_status_read()
    s.close()
    return L, status


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_nan_level_set_on_triangles(orc, dg, p):
    wl = W.rider_kothe(n=6, p=p, elem="tri")
    Np = wl.N // 72
    w = wl.w.copy()
    w[1, 14 * Np + Np // 2] = np.nan
    pb, vc = _kin(orc, wl)
    L_ref = orc.tri_rhs(pb, vc, 0.7, w)
    L, status = _rhs(dg, wl, w)
    nan, ref = np.isnan(L), np.isnan(L_ref)
    assert ref[0].sum() == 4 * Np  # the triangle and its three neighbours
    assert np.array_equal(nan[0], ref[0])
    # (the edges read psi at their own nodes alone, the oracle at all of the element's)
    assert nan[1].any() and not (nan[1] & ~ref[1]).any()
    assert status == -5  # DG_ERR_NONFINITE


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
def test_nan_level_set_on_rectangles(dg, p):
    wl = W.rider_kothe(n=6, p=p)
    Np = (p + 1) ** 2
    w = wl.w.copy()
    w[1, 14 * Np + Np // 2] = np.nan
    L, status = _rhs(dg, wl, w)
    L0, _ = _rhs(dg, wl, wl.w.copy())
    assert np.isfinite(L[0]).all() and np.isnan(L[1]).any()
    far = np.ones(wl.N, bool)  # elements that neither hold nor touch the node
    for e in (14, 13, 15, 8, 20):
        far[e * Np:(e + 1) * Np] = False
    assert np.array_equal(L[:, far], L0[:, far])
    assert status == -5

"""Triangle groups chosen by the mesh (pick_tri_epb, csrc/dg_tri.cuh): right-hand sides against the oracle
on meshes of few triangles per SM (groups of one up), of one group per SM and of several, with a ragged last
group, within 1e-12 of the oracle's scale, as tests/test_gpu_triangles.py holds the same sums."""
import numpy as np
import pytest

from paper_2306_05002_gb300 import workloads as W
from tests.test_gpu_triangles import _broken, _kin

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [3, 13, 27, 33, 49])
def test_tri_rhs_by_group_size(orc, dg, p, n):
    import torch
    wl = W.rider_kothe(n=n, p=p, elem="tri")
    w = _broken(wl, p)
    pb, vc = _kin(orc, wl)
    s = dg.KinematicSolver(wl)
    L_ref, S = orc.tri_rhs(pb, vc, 0.7, w, want_scale=True)
    L = s.dg_kin_rhs(torch.from_numpy(w.copy()).cuda(), 0.7).cpu().numpy()
    for v in range(2):
        assert np.abs(L[v] - L_ref[v]).max() <= 1e-12 * S[v].max(), v
    assert s.dg_status_read() == 0
    s.close()

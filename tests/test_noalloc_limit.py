"""The size limit of dg_rhs_noalloc: a call is held to a 256-byte status line, the operator table
without its derived part, 7 fields per node and 14 trace fields per face node (17 with viscous stress)
in DG_NOALLOC_SCRATCH_BYTES.  The largest mesh of a column of elements runs and equals dg_rhs; one
element more is refused before any GPU work."""
import ctypes

import numpy as np
import pytest

from paper_2306_05002_gb300 import workloads as W
from tests.test_zz_no_alloc import _entry, _noalloc_vs_rhs, _structs


def _largest(p, viscous):
    P1, cap, al = p + 1, 32 << 20, lambda b: (b + 255) // 256 * 256
    ops = al(8 * (4 * P1 * P1 + 3 * P1 + P1 * P1))
    need = lambda E: 256 + ops + al(56 * E * P1 * P1) + 8 * (17 if viscous else 14) * E * 4 * P1
    E = 1
    while need(E + 1) <= cap:
        E += 1
    return E


CASES = [(p, v) for p in (1, 3, 5) for v in (False, True)]


@pytest.mark.parametrize("p,viscous", CASES)
def test_one_element_more_is_refused(p, viscous):
    pkg, f = _entry()
    wl = W.Workload(name="big", dim=2, nx=1, ny=_largest(p, viscous) + 1, p=p, viscous=viscous)
    m, p, e, Gamma, eps, o = _structs(pkg, wl)
    assert f(ctypes.byref(m), p, ctypes.byref(e), 1.0, 0.01, ctypes.byref(o), ctypes.c_void_p(16),
             ctypes.c_void_p(32), None) == -1  # DG_ERR_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("p,viscous", CASES)
def test_the_largest_mesh_runs(dg, p, viscous):
    import torch
    pkg, f = _entry()
    ny = _largest(p, viscous)
    nx = next(d for d in range(int(ny ** 0.5), 0, -1) if ny % d == 0)
    wl = W.rayleigh_taylor(n=4, p=p, seed=3)
    big = W.Workload(**wl.problem_kwargs(), name="limit")
    big.nx, big.ny, big.viscous, big.surface_tension = nx, ny // nx, viscous, False
    x, y = W.node_coords(big)
    d = 0.2 * (big.y1 - big.y0)
    phi = 0.5 + 0.4 * np.tanh((y - 0.5 * (big.y0 + big.y1)) / d)
    big.w = W.conserved(big, phi, d * np.log(phi / (1 - phi)), 1e5, 0.3 * np.sin(x), 0.2 * np.cos(y))
    _noalloc_vs_rhs(pkg, f, big, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))

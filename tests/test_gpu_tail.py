"""The single-CTA tail against the grid kernels it replaces, bit for bit.

The tail runs the small levels' steps with the grid kernels' expressions on
the same operands in the same order, so the iterate after any number of
cycles is the same whatever level it starts at.  Covered here: the paper's
smoother and transfers (every pairing), weighted Jacobi with odd and even
sweep counts (the iterate ends in either buffer), truncated hierarchies (a
coarsest grid of several unknowns), and the smallest grids, which are all tail.
"""
import os

import numpy as np
import pytest

from paper_1208_4247_gb300 import inputs

pytestmark = pytest.mark.gpu


def cycles(monkeypatch, tail_n, d, n, kw, count=3):
    import torch
    from paper_1208_4247_gb300 import build
    from paper_1208_4247_gb300.gmg import Solver
    build.build()
    monkeypatch.setenv("GMG_TAIL_N", str(tail_n))
    f = torch.from_numpy(inputs.rhs_uniform(d, n, 11)).cuda()
    u = torch.from_numpy(inputs.rhs_uniform(d, n, 12)).cuda()
    with Solver(d, n, **kw) as S:
        rel = S.cycles(f, u, count)
    return u.cpu().numpy(), rel


CASES = [
    (2, 64, dict(smoother="mcgs", transfer="paper", nu1=1, nu2=2)),
    (2, 32, dict(smoother="mcgs", transfer="fw", nu1=2, nu2=1)),
    (2, 64, dict(smoother="rbgs", transfer="paper", nu1=2, nu2=2)),
    (2, 4, dict(smoother="mcgs", transfer="paper", nu1=1, nu2=1)),
    (3, 16, dict(smoother="mcgs", transfer="paper", nu1=1, nu2=2)),
    (3, 8, dict(smoother="mcgs", transfer="fw", nu1=1, nu2=1)),
    (3, 32, dict(smoother="wjacobi", transfer="paper", nu1=2, nu2=1)),
    (2, 64, dict(smoother="wjacobi", nu1=1, nu2=2)),
    (2, 32, dict(smoother="wjacobi", nu1=3, nu2=0, levels=3)),
    (3, 16, dict(smoother="rbgs", nu1=0, nu2=2, levels=2, coarse_sweeps=5)),
]


@pytest.mark.parametrize("d,n,kw", CASES)
def test_tail_equals_grid_kernels(monkeypatch, d, n, kw):
    pytest.importorskip("torch")
    ref, rel_ref = cycles(monkeypatch, 1, d, n, kw)  # every level on grid kernels
    for tail_n in (0, n):  # the default threshold, the whole hierarchy
        u, rel = cycles(monkeypatch, tail_n, d, n, kw)
        assert np.array_equal(u, ref), (tail_n, np.max(np.abs(u - ref)))
        assert rel == rel_ref

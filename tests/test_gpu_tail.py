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
    if tail_n == 1:  # every level on grid kernels
        monkeypatch.setenv("GMG_FUSED_LEGS", "0")
    else:
        monkeypatch.delenv("GMG_FUSED_LEGS", raising=False)
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


SLAB = [(n, prec, dict(nu1=nu1, nu2=nu2, **kw))
        for prec in ("fp64", "df", "fp32", "bf16")
        for n, nu1, nu2, kw in ((64, 2, 2, {}), (32, 1, 3, {}), (16, 2, 1, {}), (32, 2, 2, {"levels": 4}),
                                (16, 1, 1, {"levels": 3}), (64, 1, 2, {"levels": 5, "coarse_sweeps": 3}))]
SLAB += [(32, "fp64", dict(nu1=0, nu2=2)), (16, "fp64", dict(nu1=2, nu2=0)),
         (32, "fp64", dict(nu1=1, nu2=2, cycle="fmg")), (16, "fp64", dict(nu1=2, nu2=2, cycle="fmg")),
         (32, "df", dict(nu1=0, nu2=1)), (64, "fp32", dict(nu1=2, nu2=0))]


@pytest.mark.parametrize("n,prec,kw", SLAB)
def test_slab_tail_equals_grid_kernels(monkeypatch, n, prec, kw):
    """The cluster of 16 CTAs (levels 33^3 and 17^3 in distributed shared
    memory) against the grid kernels, bit for bit: as the tail of a larger
    hierarchy and as the whole of a small one, hierarchies cut below 9^3,
    no pre- or post-smoothing (full residual, full prolongation), FMG."""
    pytest.importorskip("torch")
    kw = dict(kw, precision=prec)
    if prec != "fp64":
        kw["inner_cycles"] = 2 if prec == "fp32" else 1
    ref, rel_ref = cycles(monkeypatch, 1, 3, n, kw)
    u, rel = cycles(monkeypatch, 0, 3, n, kw)
    assert np.array_equal(u, ref), np.max(np.abs(u - ref))
    assert rel == rel_ref


LEGS = [(n, dict(smoother=sm, transfer=tr, nu1=nu1, nu2=nu2, **kw))
        for sm, tr, nu1, nu2, kw in (
            ("wjacobi", "fw", 2, 2, {}), ("wjacobi", "paper", 1, 3, {}), ("rbgs", "fw", 2, 2, {}),
            ("rbgs", "fw", 1, 3, {"cycle": "fmg"}), ("rbgs", "paper", 3, 1, {}),
            ("mcgs", "paper", 1, 1, {}), ("mcgs", "fw", 2, 1, {}), ("mcgs", "paper", 1, 2, {"cycle": "fmg"}))
        for n in (32, 64, 128, 256, 512)]
LEGS += [(1024, dict(smoother="mcgs", transfer="paper", nu1=1, nu2=1)),
         (128, dict(smoother="wjacobi", nu1=6, nu2=6)), (64, dict(smoother="rbgs", nu1=2, nu2=2, levels=1)),
         (64, dict(smoother="rbgs", nu1=2, nu2=2, levels=2, coarse_sweeps=7))]


@pytest.mark.parametrize("n,kw", LEGS)
def test_legs_2d_equal_grid_kernels(monkeypatch, n, kw):
    """The 2D leg kernels (a level's down and up half as one launch each,
    halos computed again) against a launch per step, bit for bit: every tile
    size, each smoother with odd and even step counts, both transfers, the
    first cycle a full-multigrid pass, hierarchies cut short."""
    pytest.importorskip("torch")
    ref, rel_ref = cycles(monkeypatch, 1, 2, n, kw)
    u, rel = cycles(monkeypatch, 0, 2, n, kw)
    assert np.array_equal(u, ref), np.max(np.abs(u - ref))
    assert rel == rel_ref

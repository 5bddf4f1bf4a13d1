"""The 3D outer residual of FP32 / BF16 refinement (6 sigma = 6 q + (sum - 6 u),
divided on the FP32 pipe) by row kernels (n < 128) and walkers, against the
oracle: the reported norms are the iterate's, and refinement gets down to the
FP64 rounding of u.

Tolerances: sigma carries a few roundings of sum and u, each at most 2^-53 *
6 |u|, with |u| <= |f| / (3 pi^2) against b = |f| / n^2: 12 * 2^-53 * n^2 / 30 of
the starting residual, 3e-13 at n = 128 (taken twice); the norm of a residual far
above that agrees to 1e-10."""
import numpy as np
import pytest

import oracle
from paper_1208_4247_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [("fp32", 8), ("fp32", 64), ("fp32", 128), ("bf16", 32),
                                    ("bf16", 128)])
def test_refinement_to_the_rounding_of_u(prec, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_4247_gb300 import build
    from paper_1208_4247_gb300.gmg import Solver
    build.build()
    f = inputs.rhs_uniform(3, n, 13)
    b = oracle.scale_rhs(f)
    b0 = oracle.norm2(oracle.residual(b, np.zeros_like(f)))
    fd, floor = torch.from_numpy(f).cuda(), 2 * 12 * 2.0 ** -53 * n * n / 30 + 1e-14
    with Solver(3, n, precision=prec, inner_cycles=2 if prec == "fp32" else 1) as S:
        for steps in (2, 30):
            u = torch.zeros_like(fd)
            rel = S.cycles(fd, u, steps)[-1]
            ref = oracle.norm2(oracle.residual(b, u.cpu().numpy())) / b0
            assert abs(rel - ref) <= 1e-10 * ref + floor, (steps, rel, ref)
    assert ref <= floor

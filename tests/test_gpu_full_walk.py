"""The 3D FP64 levels whose full residual, stored norm and full restriction run
by walkers (n >= 128: no red-black colour is zero before the restriction, or
the smoother is learned), against the CPU oracle.

Tolerances: a cycle 1e-12 of u (the form's bar; the restriction sums the same
terms in another order, a few 2^-53 of them); a norm 1e-10 (millions of squares
in two orders, 2^-53 times the adds of one partial sum's chain)."""
import numpy as np
import pytest

import oracle
from paper_1208_4247_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_4247_gb300 import build
    build.build()
    return torch


def start(n):
    u = np.zeros((n + 1,) * 3)
    u[1:-1, 1:-1, 1:-1] = np.random.default_rng(31).standard_normal((n - 1,) * 3)
    return inputs.rhs_uniform(3, n, 9), u


@pytest.mark.parametrize("n,sm,om,nu1,nu2", [(128, "wjacobi", 6 / 7, 2, 2),
                                             (256, "wjacobi", 6 / 7, 1, 1),
                                             (128, "rbgs", 0.8, 0, 2)])
def test_cycle_parity(torch_cuda, n, sm, om, nu1, nu2):
    from paper_1208_4247_gb300.gmg import Solver
    f, u = start(n)
    cfg = oracle.make_cfg(3, n, 0, oracle.RBGS if sm == "rbgs" else oracle.WJACOBI, om, nu1, nu2, 1)
    b, uo = oracle.scale_rhs(f), u.copy()
    oracle.vcycle(cfg, b, uo)
    ud = torch_cuda.from_numpy(u).cuda()
    with Solver(3, n, smoother=sm, omega=om, nu1=nu1, nu2=nu2) as S:
        rel = S.cycles(torch_cuda.from_numpy(f).cuda(), ud, 1)[0]
    ug = ud.cpu().numpy()
    assert np.linalg.norm(ug - uo) <= 1e-12 * np.linalg.norm(uo)
    assert np.max(np.abs(ug - uo)) <= 1e-12 * np.max(np.abs(uo))
    assert rel == pytest.approx(oracle.norm2(oracle.residual(b, ug)) /
                                oracle.norm2(oracle.residual(b, u)), rel=1e-10)


@pytest.mark.parametrize("n", [128, 256])
def test_learned_norms(torch_cuda, n):
    """Norms of iterates whose residual the learned smoother then takes."""
    from paper_1208_4247_gb300.gmg import Solver, jacobi_weights
    f, u = start(n)
    b = oracle.scale_rhs(f)
    ud = torch_cuda.from_numpy(u).cuda()
    with Solver(3, n, smoother="learned", nu1=1, nu2=1) as S:
        for level in range(n.bit_length() - 3):
            S.set_learned_weights(level, jacobi_weights(3, 6 / 7))
        rel = S.cycles(torch_cuda.from_numpy(f).cuda(), ud, 2)
    assert rel[0] > rel[1]
    assert rel[1] == pytest.approx(oracle.norm2(oracle.residual(b, ud.cpu().numpy())) /
                                   oracle.norm2(oracle.residual(b, u)), rel=1e-10)

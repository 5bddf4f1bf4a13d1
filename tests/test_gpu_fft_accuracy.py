"""Accuracy of the direct solve where its eliminations could lose it, and at the
largest sizes (the 512-thread tiles), in units u = 2^-53.

A step of an elimination has two rounded operations, of RMS at most u / sqrt(3)
each; an error decays by r per step (r + 1/r = 2 + lambda of the line), so that
about min(n/2, 1 / (2 (1 - r))) steps count, twice two sweeps of them.  The
transforms and the reference add a few u, taken as 16.  Twice the RMS is allowed.

A mode whose coefficients c_k have reached their limit r shares the rounding of r
along the whole line: kept as c_k in double it would enter the solution 2 / (1 -
r) times over, 40 to 80 u for the modes here."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_4247_gb300 import build
    build.build()
    return torch


def tolerance(steps):
    return U * (16 + 2 * np.sqrt(4 * 2 * steps / 3))


def sine(torch, k, n):
    """sin(pi k j / n) from an angle of the first quadrant, in extended precision"""
    j = np.arange(n + 1, dtype=np.int64) * k % (2 * n)
    a = np.where(j > n, j - n, j)
    a = np.minimum(a, n - a).astype(np.longdouble)
    s = np.sin(a * (4 * np.arctan(np.longdouble(1)) / n)).astype(np.float64)
    return torch.from_numpy(np.where(j > n, -s, s)).cuda()


def eigenvalue(k, n):
    return 4 * np.sin(2 * np.arctan(np.longdouble(1)) * k / n) ** 2


@pytest.mark.parametrize("n,k", [(4096, 20), (4096, 21), (8192, 23), (8192, 31)])
def test_modes_whose_coefficients_share_a_rounding(torch_cuda, n, k):
    torch = torch_cuda
    from paper_1208_4247_gb300.gmg import FFTSolver
    phi = sine(torch, 1, n)[:, None] * sine(torch, k, n)  # x is the last axis
    lam = eigenvalue(k, n)
    ref = phi / float(lam + eigenvalue(1, n))
    f, u = phi * float(n) ** 2, torch.zeros_like(phi)
    with FFTSolver(2, n) as F:
        F.solve(f, u)
    gap = float(np.sqrt(lam + lam * lam / 4) - lam / 2)  # 1 - r
    assert float((u - ref).norm() / ref.norm()) <= tolerance(1 / (2 * gap))


def residual(torch, f, u):
    """h^2 f - A'u of the interior, summed in pairs of doubles"""
    d, n = f.dim(), f.shape[0] - 1
    c = (slice(1, -1),) * d
    s, e = f[c] / n ** 2, torch.zeros_like(f[c])  # (a power of two)

    def add(s, e, b):
        t = s + b
        z = t - s
        return t, e + ((s - (t - z)) + (b - z))

    for _ in range(d):
        s, e = add(s, e, -2.0 * u[c])
    for ax in range(d):
        for sl in (slice(0, -2), slice(2, None)):
            i = list(c)
            i[ax] = sl
            s, e = add(s, e, u[tuple(i)])
    return s + e


@pytest.mark.parametrize("d,n", [(2, 256), (2, 2048), (2, 4096), (2, 8192), (3, 64), (3, 256), (3, 512)])
def test_error_of_a_rough_right_hand_side(torch_cuda, d, n):
    """The error is the correction that its residual asks for."""
    torch = torch_cuda
    from paper_1208_4247_gb300.gmg import FFTSolver
    g = torch.Generator(device="cuda").manual_seed(n)
    f = torch.rand((n + 1,) * d, generator=g, dtype=torch.float64, device="cuda") * 2 - 1
    u, r, du = torch.zeros_like(f), torch.zeros_like(f), torch.zeros_like(f)
    with FFTSolver(d, n) as F:
        F.solve(f, u)
        r[(slice(1, -1),) * d] = residual(torch, f, u) * float(n) ** 2
        F.solve(r, du)
    assert float(du.norm() / u.norm()) <= tolerance(n / 2)

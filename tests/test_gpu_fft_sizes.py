"""The direct sine-transform solve at every kind of size its kernels meet:
the degenerate folds (n = 2, 4), blocks that end in a radix-2, -4 or -8 stage,
one warp per pair of lines and several, a last CTA that is partly empty.

Reference: scipy's DST-I with the discrete eigenvalues.  Tolerance (relative
L2), derived: in units of 2^-53 each transform adds at most 16 per fold or
radix-2 level (2 (d-1) transforms of log2 n levels here, 2 d in the
reference), and each of the n/2 steps of the two elimination sweeps at most
two of its own (an error never grows along a sweep, the coefficients are
below 1).
"""
import numpy as np
import pytest

from paper_1208_4247_gb300 import inputs

pytestmark = pytest.mark.gpu


def reference(f):
    from scipy.fft import dstn
    d, n = f.ndim, f.shape[0] - 1
    inner = (slice(1, -1),) * d
    lam = 4 * np.sin(np.arange(1, n) * (np.pi / (2 * n))) ** 2
    tot = lam
    for _ in range(d - 1):
        tot = tot[..., None] + lam
    u = np.zeros_like(f)
    c = dstn(f[inner] / n ** 2, type=1, norm="ortho") / tot
    u[inner] = dstn(c, type=1, norm="ortho")
    return u


@pytest.mark.parametrize("d,n", [(2, 2 ** k) for k in range(1, 12)] +
                         [(3, 2 ** k) for k in range(1, 9)])
def test_every_size(d, n):
    torch = pytest.importorskip("torch")
    pytest.importorskip("scipy")
    from paper_1208_4247_gb300 import build
    from paper_1208_4247_gb300.gmg import FFTSolver
    build.build()
    f = inputs.rhs_uniform(d, n, 7 + n)
    ref = reference(f)
    fd = torch.from_numpy(f).cuda()
    fd[(0,) * d] = 3.0  # boundary values of f are not read into the solution
    u = torch.full_like(fd, 5.0)  # every node of u is written
    with FFTSolver(d, n) as F:
        F.solve(fd, u)
        first = u.cpu().numpy()
        F.solve(fd, fd)  # in place
    tol = 2.0 ** -53 * (16 * (4 * d - 2) * np.log2(n) + 2 * n)
    assert np.linalg.norm(first - ref) <= tol * np.linalg.norm(ref)
    edge = np.ones_like(f, bool)
    edge[(slice(1, -1),) * d] = False
    assert not np.any(first[edge])
    assert np.array_equal(fd.cpu().numpy(), first)

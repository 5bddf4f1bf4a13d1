"""One refinement step of a batch whose levels take every launch shape of the
legs (parts of a warp, one tile, several tiles, rows wider than a warp) against
the same cycles in FP64 numpy, with the kernels' FP32 constants 1/(2d) and
omega (the coarse solve amplifies the offset of fl(1/6) by 1/lambda_min).

Tolerance: a node's value passes through at most 10 levels of about 40 rounded
FP32 operations, each off by at most 2^-24 of the level's largest value:
400 * 6e-8 = 2.4e-5 of max|u|, taken as 3e-5 (BF16 storage: one rounding of
2^-9 per stored value, about 3 per level and cycle: 10 * 6 * 2e-3 = 0.12)."""
import numpy as np
import pytest

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


def nsum(u):
    d = u.ndim
    c = (slice(1, -1),) * d
    s = np.zeros_like(u[c])
    for ax in range(d):
        for sl in (slice(0, -2), slice(2, None)):
            i = list(c)
            i[ax] = sl
            s += u[tuple(i)]
    return s


def smooth(u, q, sweeps, om, rb):
    d = u.ndim
    w = float(np.float32(1 / (2 * d)))
    om = float(np.float32(om))
    c = (slice(1, -1),) * d
    par = sum(np.meshgrid(*[np.arange(1, u.shape[0] - 1)] * d, indexing="ij")) & 1
    for _ in range(sweeps):
        if rb:
            for color in (0, 1):
                u[c] = np.where(par == color, w * nsum(u) + q[c], u[c])
        else:
            u[c] += om * (w * nsum(u) + q[c] - u[c])


def vcycle(u, q, nu1, nu2, om, rb):
    d, n = u.ndim, u.shape[0] - 1
    c = (slice(1, -1),) * d
    if n == 2:
        u[c] = q[c]
        return
    smooth(u, q, nu1, om, rb)
    r = np.zeros_like(u)
    r[c] = float(np.float32(1 / (2 * d))) * nsum(u) + q[c] - u[c]
    for ax in range(d):  # full weighting, one axis after the other
        r = np.moveaxis(r, ax, 0)
        w = np.zeros((n // 2 + 1,) + r.shape[1:])
        w[1:-1] = 0.25 * r[1:-2:2] + 0.5 * r[2:-1:2] + 0.25 * r[3::2]
        r = np.moveaxis(w, 0, ax)
    e = np.zeros_like(r)
    vcycle(e, 4 * r, nu1, nu2, om, rb)
    for ax in range(d):  # linear interpolation
        e = np.moveaxis(e, ax, 0)
        w = np.zeros((2 * e.shape[0] - 1,) + e.shape[1:])
        w[::2] = e
        w[1::2] = 0.5 * (e[:-1] + e[1:])
        e = np.moveaxis(w, 0, ax)
    u += e
    smooth(u, q, nu2, om, rb)


MIX = [(2, 4), (3, 4), (2, 8), (3, 8), (3, 16), (2, 64), (3, 32), (2, 128), (3, 64), (2, 256),
       (3, 128), (2, 2048), (3, 256), (2, 256), (3, 32)]


@pytest.mark.parametrize("prec,sm,nu1,nu2,k,ctas,tol", [
    ("fp32", "wjacobi", 1, 1, 2, 0, 3e-5), ("fp32", "wjacobi", 1, 1, 1, 5, 3e-5),
    ("fp32", "wjacobi", 2, 2, 1, 0, 3e-5), ("fp32", "wjacobi", 0, 2, 1, 0, 3e-5),
    ("fp32", "wjacobi", 2, 0, 1, 0, 3e-5), ("fp32", "rbgs", 1, 1, 1, 0, 3e-5),
    ("bf16", "wjacobi", 1, 1, 1, 0, 0.12)])
def test_one_step_equals_numpy(torch_cuda, prec, sm, nu1, nu2, k, ctas, tol):
    torch = torch_cuda
    from paper_1208_4247_gb300.gmg import Batch
    fs = [inputs.rhs_uniform(d, n, 60 + i) for i, (d, n) in enumerate(MIX)]
    fd = [torch.from_numpy(f).cuda() for f in fs]
    ud = [torch.zeros_like(f) for f in fd]
    with Batch([d for d, _ in MIX], [n for _, n in MIX], smoother=sm, omega=0.8, nu1=nu1, nu2=nu2,
               precision=prec, inner_cycles=k, maxit=1, ctas=ctas) as B:
        it, rel, steps, conv = B.solve(fd, ud, rtol=1e-14)
    assert steps == 1 and set(it) == {1}
    for (d, n), f, u in zip(MIX, fs, ud):
        e, q = np.zeros_like(f), f / (2 * d * n * n)
        for _ in range(k):
            vcycle(e, q, nu1, nu2, 0.8, sm == "rbgs")
        assert np.max(np.abs(u.cpu().numpy() - e)) <= tol * np.max(np.abs(e)), (d, n)

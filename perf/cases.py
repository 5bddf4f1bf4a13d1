"""The work whose speed is measured: whole calls of the public entry points.

One pass is what a program that uses the solver does again and again: a solve
of the finite-difference Poisson system on a grid from u = 0 (``Solver``, a
``Batch``, ``FFTSolver``) or one loss and gradient evaluation of the learned
smoother.  ``listed()`` names the cases, ``draw()`` gives more of the same
ranges: every grid size is a power of two (the library takes no other), so the
odd sizes are the odd sweep counts, batch counts, weights, tolerances and row
pitches.

A case is one of these kinds:

* ``solve``   -- ``Solver.solve`` / ``solve_strided`` / ``solve_host`` in one of
  the precisions, smoothers, transfers and cycles;
* ``learned`` -- ``Solver.solve`` with the convolutional smoother on every level
  with n >= 8;
* ``batch``   -- ``Batch.solve`` of a seeded mix of 2D and 3D solves;
* ``fft``     -- ``FFTSolver.solve``, the direct sine-transform solve;
* ``grad``    -- ``learned_loss_grad``, forward and backward of the training.

Iterative solves return the solution and the integers (cycles, converged).
The relative residual they also report is left out: at the stopping
tolerance it consists of the rounding errors of the solution.
"""
import numpy as np
import torch

from paper_1208_4247_gb300 import gmg

# the size classes of the batched workload (d, n)
CLASSES = [(2, 2 ** k) for k in range(6, 11)] + [(3, 2 ** k) for k in range(4, 8)]


def _solve(name, d, n, **kw):
    c = dict(kind="solve", d=d, n=n, precision="fp64", smoother="rbgs", transfer="fw", cycle="v",
             nu1=2, nu2=2, omega=0.8, inner_cycles=1, rtol=1e-10, rhs="uniform", call="device",
             pad=0)
    c.update(kw)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest solve a program makes by itself: 2D, 257^2, weighted Jacobi V(2,2)
        _solve("jacobi_2d_257", 2, 256, smoother="wjacobi", rhs="sine_uniform"),
        # a small 3D solve in the default configuration (FP64, red-black V(2,2))
        _solve("rbgs_3d_65", 3, 64),
        # the ordinary 3D solve in the default configuration
        _solve("rbgs_3d_257", 3, 256),
        # the same system in the form recommended for speed (double-float refinement)
        _solve("df_3d_257", 3, 256, precision="df"),
        # large grid, single-precision cycles in FP64 refinement
        _solve("fp32_3d_513", 3, 512, precision="fp32", inner_cycles=3, rhs="sine_gauss"),
        # BF16 storage in FP64 refinement
        _solve("bf16_3d_257", 3, 256, precision="bf16", rhs="sine_gauss"),
        # the paper's own smoother and transfers, at the paper's tolerance
        _solve("paper_2d_1025", 2, 1024, smoother="mcgs", transfer="paper", nu1=1, nu2=1,
               rtol=1e-6, rhs="sine_uniform"),
        # full multigrid as the first cycle, large 2D grid
        _solve("fmg_2d_2049", 2, 2048, cycle="fmg", nu1=1, nu2=2, rhs="sine_uniform"),
        # many solves of uneven sizes at once, at the settings the tuner picks for 512 of them
        dict(name="batch_512", kind="batch", count=512, smoother="wjacobi", omega=0.0, nu1=1,
             nu2=1, precision="fp32", inner_cycles=10, chunk=4096, ctas=2432, rtol=1e-10),
        # the learned smoother on every level, correlated right-hand side
        dict(name="learned_3d_257", kind="learned", d=3, n=256, nu1=1, nu2=1, rtol=1e-10),
        # the direct solve by sine transforms
        dict(name="fft_3d_257", kind="fft", d=3, n=256),
        # one training sample of the learned smoother: loss and weight gradient
        dict(name="grad_3d_65", kind="grad", d=3, n=64, coarse_cycles=12),
    ]


def draw(rng):
    kind = rng.choice(["solve2", "solve3", "refine", "paper", "fmg", "batch", "learned", "fft", "grad"])
    p2 = lambda lo, hi: 2 ** rng.randint(lo, hi)  # noqa: E731
    nu = dict(nu1=rng.randint(1, 3), nu2=rng.randint(1, 3))
    rtol = 10.0 ** -rng.uniform(6, 10)
    rhs = rng.choice(["uniform", "sine_uniform", "sine_gauss"])
    omega = round(rng.uniform(0.7, 0.9), 3)
    if kind in ("solve2", "solve3"):
        d = 2 if kind == "solve2" else 3
        smoother = rng.choice(["rbgs", "wjacobi"])
        n = p2(6, 11) if d == 2 else p2(4, 8)
        call = rng.choice(["device", "device", "strided", "host"])
        if call == "host":
            n = min(n, 1024 if d == 2 else 128)
        return _solve(None, d, n, smoother=smoother, rhs=rhs, omega=omega, rtol=rtol, call=call,
                      pad=rng.choice([1, 3, 8, 17]) if call == "strided" else 0, **nu)
    if kind == "refine":
        precision = rng.choice(["df", "df", "fp32", "bf16"])
        n = p2(5, 9) if precision == "fp32" else p2(5, 8)
        if precision == "bf16":
            nu = dict(nu1=2, nu2=2)
        return _solve(None, 3, n, precision=precision, rhs=rhs, rtol=rtol,
                      inner_cycles=rng.randint(2, 4) if precision == "fp32" else 1, **nu)
    if kind == "paper":
        d = rng.choice([2, 3])
        return _solve(None, d, p2(6, 12) if d == 2 else p2(4, 8), smoother="mcgs",
                      transfer="paper", rhs="sine_uniform", rtol=1e-6, **nu)
    if kind == "fmg":
        d = rng.choice([2, 3])
        return _solve(None, d, p2(6, 12) if d == 2 else p2(4, 8), cycle="fmg", rhs=rhs, rtol=rtol, **nu)
    if kind == "batch":
        return dict(kind="batch", count=int(round(2 ** rng.uniform(1.5, 8.5))),
                    smoother=rng.choice(["wjacobi", "wjacobi", "rbgs"]), omega=0.0, nu1=1, nu2=1,
                    precision="fp32", inner_cycles=rng.randint(2, 10),
                    chunk=rng.choice([0, 1024, 4096]), ctas=rng.choice([0, 1216, 2432]), rtol=rtol)
    if kind == "learned":
        d = rng.choice([2, 3, 3])
        return dict(kind="learned", d=d, n=p2(6, 10) if d == 2 else p2(5, 8), nu1=1, nu2=1, rtol=rtol)
    if kind == "fft":
        d = rng.choice([2, 3])
        return dict(kind="fft", d=d, n=p2(6, 12) if d == 2 else p2(4, 8))
    d = rng.choice([2, 3, 3])
    return dict(kind="grad", d=d, n=p2(5, 8) if d == 2 else p2(4, 6), coarse_cycles=rng.randint(8, 30))


# ------------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _inner(a):
    return a[(slice(1, -1),) * a.dim()]


def _axes(d, v):
    """prod over the d axes of the vector v (outer product)."""
    out = v
    for _ in range(d - 1):
        out = out[..., None] * v
    return out


def _rhs(d, n, kind, g):
    f = torch.zeros((n + 1,) * d, dtype=torch.float64, device="cuda")
    shape = (n - 1,) * d
    if kind == "uniform":  # i.i.d. U[-1, 1]
        _inner(f).copy_(torch.rand(shape, generator=g, dtype=torch.float64, device="cuda") * 2 - 1)
        return f
    s = torch.sin(torch.arange(1, n, dtype=torch.float64, device="cuda") * (np.pi / n))
    if kind == "correlated":  # white noise in the sine basis, amplitude 1/|k|
        k2 = torch.arange(1, n, dtype=torch.float64, device="cuda") ** 2
        tot = k2
        for _ in range(d - 1):
            tot = tot[..., None] + k2
        c = torch.randn(shape, generator=g, dtype=torch.float64, device="cuda") / tot.sqrt()
        field = _along(c, _sine(n))
        _inner(f).copy_(field / field.square().mean().sqrt())
        return f
    # a smooth source plus noise: uniform of amplitude 1e-3 or Gaussian of sigma 1e-2
    noise = (1e-3 * (torch.rand(shape, generator=g, dtype=torch.float64, device="cuda") * 2 - 1)
             if kind == "sine_uniform" else
             1e-2 * torch.randn(shape, generator=g, dtype=torch.float64, device="cuda"))
    _inner(f).copy_(d * np.pi ** 2 * _axes(d, s) + noise)
    return f


def _weights(d, g):
    """Weights of the kind training gives: two damped smoothing steps (the
    roots of the degree-2 Chebyshev polynomial on the upper half of the
    spectrum) carried by the channel pair relu(x) - relu(-x) = x, and small
    values on every other tap."""
    T, mid = gmg.learned_taps(d), gmg.learned_taps(d) // 2
    a, b = (1.733, 0.5695) if d == 3 else (1.3895, 0.5617)
    w = 0.01 * torch.randn((2, 8, T), generator=g, dtype=torch.float32, device="cuda").cpu().numpy()
    w[0, 0, mid] += 1.0
    w[0, 1, mid] -= 1.0
    step = np.zeros(T, np.float32)
    step[mid] = a + b - a * b
    for off in (1, 3, 9)[:d]:
        step[mid - off] = step[mid + off] = a * b / (2 * d)
    w[1, 0] += step
    w[1, 1] -= step
    return w


def _mix(count):
    """The grids of a batch: size classes drawn uniformly, the same ones for
    every seed of the inputs (a batch of other sizes would be another case)."""
    g = np.random.Generator(np.random.PCG64(4))
    return [CLASSES[i] for i in g.integers(0, len(CLASSES), size=count)]


def _slices(mix):
    """Start of each solve's array in one buffer (512-byte aligned, as separate
    tensors are) and the buffer's length, in doubles."""
    at, starts = 0, []
    for d, n in mix:
        starts.append(at)
        at += -(-(n + 1) ** d // 64) * 64
    return starts, at


def _views(flat, mix):
    starts, _ = _slices(mix)
    return [flat[s:s + (n + 1) ** d].view((n + 1,) * d) for s, (d, n) in zip(starts, mix)]


# -------------------------------------------------------------- preparation

def _pitched(d, n, pad):
    """A (n+1)^d view whose rows lie n + 1 + pad apart."""
    m = n + 1
    whole = torch.zeros((m,) * (d - 1) + (m + pad,), dtype=torch.float64, device="cuda")
    return whole[..., :m]


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "batch":
        mix = _mix(case["count"])
        _, length = _slices(mix)
        f, u = (torch.zeros(length, dtype=torch.float64, device="cuda") for _ in range(2))
        fs, us = _views(f, mix), _views(u, mix)
        for v, (d, n) in zip(fs, mix):
            v.copy_(_rhs(d, n, "uniform", g))
        B = gmg.Batch([d for d, _ in mix], [n for _, n in mix], smoother=case["smoother"],
                      omega=case["omega"], nu1=case["nu1"], nu2=case["nu2"],
                      precision=case["precision"], inner_cycles=case["inner_cycles"],
                      chunk=case["chunk"], ctas=case["ctas"])
        return dict(case=case, h=B, fs=fs, us=us, u=u)
    d, n = case["d"], case["n"]
    if kind == "fft":
        f = _rhs(d, n, "uniform", g)
        return dict(case=case, h=gmg.FFTSolver(d, n), f=f, u=torch.zeros_like(f))
    if kind == "grad":
        return dict(case=case, e0=_rhs(d, n, "uniform", g), w=_weights(d, g))
    if kind == "learned":
        f = _rhs(d, n, "correlated", g)
        S = gmg.Solver(d, n, smoother="learned", nu1=case["nu1"], nu2=case["nu2"])
        w = _weights(d, g)
        for level in range(n.bit_length() - 3):  # n, n/2, ..., 8
            S.set_learned_weights(level, w)
        return dict(case=case, h=S, f=f, u=torch.zeros_like(f))
    f = _rhs(d, n, case["rhs"], g)
    S = gmg.Solver(d, n, smoother=case["smoother"], omega=case["omega"], nu1=case["nu1"],
                   nu2=case["nu2"], precision=case["precision"],
                   inner_cycles=case["inner_cycles"], cycle=case["cycle"],
                   transfer=case["transfer"])
    u = torch.zeros_like(f)
    if case["call"] == "strided":
        fp, u = _pitched(d, n, case["pad"]), _pitched(d, n, case["pad"])
        fp.copy_(f)
        f = fp
    if case["call"] == "host":
        f, u = f.cpu().pin_memory(), u.cpu().pin_memory()
    return dict(case=case, h=S, f=f, u=u)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "grad":
        loss, grad = gmg.learned_loss_grad(state["w"], state["e0"], case["coarse_cycles"])
        return loss, grad
    u = state["u"]
    if kind == "fft":
        state["h"].solve(state["f"], u)
        return u
    u.zero_()
    if kind == "batch":
        cycles, _, _, done = state["h"].solve(state["fs"], state["us"], case["rtol"])
        return u, np.array(cycles), done
    S = state["h"]
    if kind == "learned" or case["call"] == "device":
        cycles, _, done = S.solve(state["f"], u, case["rtol"])
    elif case["call"] == "strided":
        cycles, _, done = S.solve_strided(state["f"], u, case["rtol"])
    else:
        cycles, _, done = S.solve_host(state["f"].numpy(), u.numpy(), case["rtol"])
    return u, cycles, done


def work(case):
    """Right-hand side read once, solution written once; operations: one
    evaluation of the residual (a solver can do no less).  A gradient reads
    the error sample and evaluates both convolutions twice forward and once
    backward for each."""
    if case["kind"] == "batch":
        grids = _mix(case["count"])
    else:
        grids = [(case["d"], case["n"])]
    nodes = sum((n - 1) ** d for d, n in grids)
    if case["kind"] == "grad":
        return {"bytes": 8 * nodes, "flops": nodes * 2 * 16 * gmg.learned_taps(case["d"]) * 6}
    return {"bytes": 16 * nodes, "flops": sum((2 * d + 2) * (n - 1) ** d for d, n in grids)}


# -------------------------------------------------------- values in 64 bits

def _sine(n):
    """The orthonormal sine matrix (symmetric, its own inverse)."""
    k = torch.arange(1, n, dtype=torch.int64, device="cuda")
    # sin(pi j k / n) from the reduced product, so that large j k lose nothing
    return torch.sin((k[:, None] * k % (2 * n)).double() * (np.pi / n)) * (2.0 / n) ** 0.5


def _along(x, m):
    """The matrix m applied along every axis of x."""
    for a in range(x.dim()):
        x = torch.movedim(torch.tensordot(m, x, dims=([1], [a])), 0, a)
    return x


def _poisson(x):
    """A'^-1 x on the interior: A' the unscaled 5- / 7-point operator."""
    d, n = x.dim(), x.shape[0] + 1
    s = _sine(n)
    lam = 4 * torch.sin(torch.arange(1, n, dtype=torch.float64, device="cuda") * (np.pi / (2 * n))) ** 2
    tot = lam
    for _ in range(d - 1):
        tot = tot[..., None] + lam
    return _along(_along(x, s) / tot, s)


def _solution(f):
    """The solution of A'u = h^2 f on all nodes."""
    u = torch.zeros_like(f)
    n = f.shape[0] - 1
    _inner(u).copy_(_poisson(_inner(f).contiguous() / n ** 2))
    return u


def _loss_grad(e0, w):
    """The two-grid contraction loss ||S CG S e||^2 / ||e||^2 and its gradient
    in the BF16-rounded weights, coarse system solved exactly."""
    d, n = e0.dim(), e0.shape[0] - 1
    w = torch.from_numpy(w).cuda().bfloat16().double().requires_grad_(True)
    conv = torch.nn.functional.conv3d if d == 3 else torch.nn.functional.conv2d
    ident = torch.eye(n - 1, dtype=torch.float64, device="cuda")
    T = 2 * ident - torch.diag_embed(torch.ones(n - 2, dtype=torch.float64, device="cuda"), 1) \
        - torch.diag_embed(torch.ones(n - 2, dtype=torch.float64, device="cuda"), -1)
    P = torch.zeros((n - 1, n // 2 - 1), dtype=torch.float64, device="cuda")
    for j in range(n // 2 - 1):
        P[2 * j, j], P[2 * j + 1, j], P[2 * j + 2, j] = 0.5, 1.0, 0.5

    def apply(x):
        return sum(torch.movedim(torch.tensordot(T, x, dims=([1], [a])), 0, a) for a in range(d))

    def smooth(x):
        k = (8, 1) + (3,) * d, (1, 8) + (3,) * d
        z = torch.relu(conv((apply(x) / (2 * d))[None, None], w[0].reshape(k[0]), padding=1))
        return x - conv(z, w[1].reshape(k[1]), padding=1)[0, 0]

    x0 = _inner(e0).contiguous()
    x = smooth(x0)
    x = x - _along(_poisson(4 * _along(apply(x), P.t() / 2)), P)
    x = smooth(x)
    loss = x.square().sum() / x0.square().sum()
    loss.backward()
    return loss.item(), w.grad.reshape(2, 8, -1).cpu().numpy()


def exact(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "batch":
        mix = _mix(case["count"])
        u = torch.zeros(_slices(mix)[1], dtype=torch.float64, device="cuda")
        for v, (d, n) in zip(_views(u, mix), mix):
            v.copy_(_solution(_rhs(d, n, "uniform", g)))
        return u, None, None
    d, n = case["d"], case["n"]
    if kind == "fft":
        return _solution(_rhs(d, n, "uniform", g))
    if kind == "grad":
        e0 = _rhs(d, n, "uniform", g)
        return _loss_grad(e0, _weights(d, g))
    return _solution(_rhs(d, n, case.get("rhs", "correlated"), g)), None, None

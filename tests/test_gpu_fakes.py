"""What the library does where a CUDA call answers in a way that no argument
brings about (tests/cuda_fakes.cpp), each script in a process of its own."""
import pytest

import fakes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return fakes.link(str(tmp_path_factory.mktemp("fakes") / "libgmg_fakes.so"))


def test_shared_memory_limits_do_not_depend_on_the_size(lib):
    """A kernel's shared-memory limit is one value for the process, so handles of
    different sizes on different threads cannot lower it under one another's
    launches."""
    out = fakes.run(lib, """
for d, n, kw in [(2, 512, {}), (2, 64, {}), (2, 32, dict(smoother="mcgs")), (2, 256, dict(smoother="wjacobi")),
                 (2, 8, dict(smoother="wjacobi")), (3, 16, {}), (3, 32, {}), (3, 64, dict(precision="df")),
                 (3, 16, dict(precision="df")), (3, 32, dict(precision="fp32")), (3, 16, dict(precision="fp32")),
                 (3, 8, dict(precision="bf16")), (3, 32, dict(precision="bf16")), (3, 8, dict(smoother="wjacobi")),
                 (3, 4, dict(smoother="wjacobi")), (3, 128, dict(precision="fp32"))]:
    f = torch.from_numpy(inputs.rhs_uniform(d, n, 5)).cuda()
    with gmg.Solver(d, n, **kw) as S:
        S.cycles(f, torch.zeros_like(f), 1)
for d, n in [(3, 128), (3, 16), (2, 512), (2, 1024)]:
    f = torch.from_numpy(inputs.rhs_uniform(d, n, 5)).cuda()
    with gmg.FFTSolver(d, n) as F:
        F.solve(f, torch.zeros_like(f))
for k in (1, 2):
    with gmg.Batch([3, 2], [16 * k, 64 * k]) as B:
        pass
print(fake.fake_attribute_changes())
""")
    assert out == ["0"]


def test_no_room_for_a_cluster(lib):
    """Where the device cannot place a cluster of 16 CTAs the small levels run in
    the single-CTA tail: every form solves, with the same bits."""
    out = fakes.run(lib, """
for kw in (dict(), dict(precision="df"), dict(precision="fp32"), dict(precision="bf16"),
           dict(smoother="learned")):
    f = torch.from_numpy(inputs.rhs_uniform(3, 64, 6)).cuda()
    got = []
    for limit in (16, 8):
        fake.fake_cluster_limit(limit)
        u = torch.zeros_like(f)
        with gmg.Solver(3, 64, **kw) as S:
            S.set_timing(True)
            S.cycles(f, u, 2)
            tails = sorted((r["kernel"], r["level"]) for r in S.timing_report()[0] if "tail" in r["kernel"])
        got.append((u, tails))
    print(torch.equal(got[0][0], got[1][0]), got[0][1] != got[1][1])
""")
    assert out == ["True True"] * 5


def test_training_reports_a_failed_launch(lib):
    """A launch that fails inside the coarse solves of a loss, a gradient or a
    training run comes back as an error, not as a number; the next call works."""
    out = fakes.run(lib, """
w = np.random.default_rng(0).normal(0, 0.01, (2, 8, 27)).astype(np.float32)
e = torch.from_numpy(inputs.rhs_uniform(3, 64, 7)).cuda()
print("ok", gmg.learned_loss_grad(w, e, 8)[0] > 0.0)
fake.fake_cluster_fails(1)
for call in (lambda: gmg.learned_loss_grad(w, e, 8),
             lambda: gmg.learned_train(3, 64, 2, 1, w, coarse_cycles=8)):
    try:
        call()
        print("returned")
    except gmg.GMGError as ex:
        print(gmg.STATUS[ex.status])
fake.fake_cluster_fails(0)
print("ok", gmg.learned_loss_grad(w, e, 8)[0] > 0.0)
""")
    assert out == ["ok True", "ERR_CUDA", "ERR_CUDA", "ok True"]


def test_batch_tables_hold_what_the_cycle_takes(lib):
    """The chunks of the plain sweeps belong to batches that sweep outside the
    legs: V(1,1) weighted Jacobi, all of whose sweeps are the legs', is made
    without them."""
    out = fakes.run(lib, """
fake.fake_copied_bytes.restype = ctypes.c_size_t
got = []
for nu in (1, 2):
    a = fake.fake_copied_bytes()
    with gmg.Batch([2, 3], [512, 64], nu1=nu, nu2=nu):
        got.append(fake.fake_copied_bytes() - a)
# the finest levels: 511 rows of 128 groups of 4 nodes, 63 * 63 rows of 16, in items
# (24 bytes) of 256 groups
print(got[0] > 0, got[1] - got[0] >= (511 * 128 + 63 * 63 * 16) // 256 * 24)
""")
    assert out == ["True True"]


def test_direct_solver_takes_one_octant_of_sines(lib):
    """The angles of a plan's table are those of one octant, n/4 + 1 of them (a
    sine and a cosine each, in software on Arm)."""
    out = fakes.run(lib, """
fake.fake_long_sines.restype = ctypes.c_size_t
for d, n in [(2, 4096), (3, 64), (2, 4), (2, 2)]:
    a = fake.fake_long_sines()
    with gmg.FFTSolver(d, n):
        print(0 < fake.fake_long_sines() - a <= 2 * (n // 4 + 1))
""")
    assert out == ["True"] * 4

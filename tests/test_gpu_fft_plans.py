"""Direct solvers of different sizes alive at once: creating one changes nothing
for another, whichever of them is the larger (their kernels share a
shared-memory limit).  Same right-hand side, same bits before and after."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first,second", [((3, 256), (3, 64)), ((3, 128), (3, 256)),
                                          ((2, 64), (2, 2)), ((2, 16), (3, 256)),
                                          ((2, 8192), (2, 4096)), ((2, 512), (2, 8192))])
def test_a_second_plan_leaves_the_first_alone(first, second):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_4247_gb300 import build
    from paper_1208_4247_gb300.gmg import FFTSolver
    build.build()
    g = torch.Generator(device="cuda").manual_seed(3)

    def rhs(d, n):
        return torch.rand((n + 1,) * d, generator=g, dtype=torch.float64, device="cuda") * 2 - 1

    fa, fb = rhs(*first), rhs(*second)
    before, after, other = torch.zeros_like(fa), torch.zeros_like(fa), torch.zeros_like(fb)
    with FFTSolver(*first) as A:
        A.solve(fa, before)
        with FFTSolver(*second) as B:
            A.solve(fa, after)
            B.solve(fb, other)
            again = torch.zeros_like(fb)
            A.solve(fa, after)
            B.solve(fb, again)
    assert torch.equal(before, after)
    assert torch.equal(other, again)
    assert bool(torch.isfinite(before).all()) and float(before.abs().max()) > 0.0

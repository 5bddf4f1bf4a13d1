"""A solve of a batch gives the same bits however its levels are cut into tiles:
alone (many short walks), among many others (few long ones) and on few CTAs.
Each node's value is formed from the same operands in the same order in every
cut, so a wrong operand at a tile's edge shows as a difference."""
import pytest

from paper_1208_4247_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("sm,nu", [("wjacobi", (1, 1)), ("wjacobi", (2, 2)), ("rbgs", (1, 1))])
def test_same_bits_in_every_tiling(prec, sm, nu):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_4247_gb300 import build
    from paper_1208_4247_gb300.gmg import Batch
    build.build()
    sizes = [(3, 256), (3, 128), (3, 32), (2, 1024), (2, 256), (2, 16)]
    fs = [torch.from_numpy(inputs.rhs_uniform(d, n, 80 + i)).cuda() for i, (d, n) in enumerate(sizes)]

    def solve(mix, ctas=0):
        us = [torch.zeros_like(fs[i]) for i in mix]
        with Batch([sizes[i][0] for i in mix], [sizes[i][1] for i in mix], smoother=sm, omega=0.8,
                   nu1=nu[0], nu2=nu[1], precision=prec, inner_cycles=2, maxit=2, ctas=ctas) as B:
            B.solve([fs[i] for i in mix], us, rtol=1e-14)
        return us

    ref = solve(range(len(sizes)))
    for i in range(len(sizes)):
        assert torch.equal(solve([i])[0], ref[i]), sizes[i]
    for j, u in enumerate(solve(list(range(len(sizes))) * 5, ctas=37)):
        assert torch.equal(u, ref[j % len(sizes)]), sizes[j % len(sizes)]

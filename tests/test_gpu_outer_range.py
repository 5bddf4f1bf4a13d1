"""FP32 / BF16 refinement in 3D near the ends of the FP32 range.  Scaling f by a
power of two scales every operation of a solve exactly as long as the inner
values stay normal FP32 numbers, so the solution has to be the scaled one, bit
for bit, up to a sigma of h^2 f / 6 that FP32 itself holds.

f is one node's value: u is largest there, 1.52 sigma, and a node's neighbours
sum to 6 x 0.52 sigma, below FLT_MAX for the sigma taken here (0.21 FLT_MAX)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [("fp32", 16), ("fp32", 128), ("bf16", 16), ("bf16", 128)])
def test_scaled_right_hand_side(prec, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_4247_gb300 import build
    from paper_1208_4247_gb300.gmg import Solver
    build.build()
    f = torch.zeros((n + 1,) * 3, dtype=torch.float64, device="cuda")
    top = 0.21 * float(np.finfo(np.float32).max)  # 6 sigma = 1.26 FLT_MAX
    shift = 2.0 ** 100
    f[(n // 2 + 1,) * 3] = top * 6 * n * n
    out = []
    for scale in (1.0, 1.0 / shift):
        u = torch.zeros_like(f)
        with Solver(3, n, precision=prec, inner_cycles=2 if prec == "fp32" else 1) as S:
            cycles, rel, done = S.solve(f * scale, u, 1e-6)
        assert done
        out.append((u / scale, cycles))
    assert out[0][1] == out[1][1]
    assert torch.equal(out[0][0], out[1][0])

"""A batch holds per level what its cycle reads: the iterate (two buffers for
weighted Jacobi), the right-hand side, and the FP64 right-hand side of the
finest level.  Margin: 24 MB for the tables, row padding (8 in 257 elements per
row) and the allocator's 2 MB granularity."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("smoother,prec,arrays", [("wjacobi", "fp32", 3), ("rbgs", "fp32", 2),
                                                  ("wjacobi", "bf16", 3)])
def test_device_memory_of_a_batch(smoother, prec, arrays):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_4247_gb300 import build
    from paper_1208_4247_gb300.gmg import Batch
    build.build()
    n, count = 256, 4
    with Batch([3], [8], smoother=smoother, precision=prec):  # loads the kernels
        pass
    free = torch.cuda.mem_get_info()[0]
    with Batch([3] * count, [n] * count, smoother=smoother, precision=prec):
        used = free - torch.cuda.mem_get_info()[0]
    elem = 4 if prec == "fp32" else 2
    levels = sum((n // 2 ** k + 1) ** 3 for k in range(8))
    need = count * (arrays * elem * levels + 8 * (n + 1) ** 3)
    assert used <= 1.04 * need + 24e6, (used, need)

"""GPU: the timing of the kernels that a call of several TV iterations spends its time
in names them, covers the benchmark's byte counts, and advances the iterate as
iterations do."""

import numpy as np
import pytest

from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,K,names,extra", [
    (512, 256, 4, {"tv_col_solve", "tv_band"}, 1), (45, 192, 4, {"tv_col_solve", "tv_band"}, 1),
    (60, 100, 3, {"tv_row_fwd", "tv_col_solve", "tv_row_inv", "tv_prox", "tv_rhs"}, 0),  # no one-kernel row half
])
def test_loop_kernel_times(H, W, K, names, extra):
    torch = need_cuda()
    import bench
    from paper_1112_1805_gb300 import binding as B
    from paper_1112_1805_gb300.api import TVSegmenter

    g = torch.Generator(device="cuda").manual_seed(W)
    f = torch.rand((H, W), device="cuda", generator=g)
    a, b = (TVSegmenter(f, np.linspace(0.1, 0.9, K)[:, None], 0.08) for _ in range(2))
    times = a.loop_kernel_times(3)
    assert set(times) == names and set(times) <= set(bench.tv_kernel_bytes(H, W, K))
    assert all(np.isfinite(t) and t >= 0 for t in times.values())
    assert int(a.get(B.SEG_ITER)) == 3 + extra
    b.step(3 + extra)
    for x in (B.SEG_U, B.SEG_W, B.SEG_BW, B.SEG_BV):
        assert torch.equal(a.get(x), b.get(x))
    a.close()
    b.close()

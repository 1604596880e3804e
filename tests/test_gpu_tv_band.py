"""GPU: several TV iterations in one call (the row half in one kernel) against the
same number of calls of one iteration (separate kernels) and the oracle: bands of
two to eight rows with a ragged last one, heights of two rows, the widths of each
row transform, periodic wrap-around at all sides, K up to 8 and past it, both
group forms, odd and even numbers of iterations (b_v's two buffers).

Both forms run the same arithmetic up to the order of a few sums, so they agree to
the oracle's bars of test_gpu_tv.py, 1e-4."""

import numpy as np
import pytest

from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu

CASES = [  # H, W, K, n, per_label
    (64, 64, 3, 12, False), (9, 48, 2, 7, False), (8, 80, 8, 6, True), (81, 96, 4, 9, False),
    (125, 128, 5, 8, False), (320, 160, 3, 5, True), (512, 256, 4, 6, False), (300, 320, 2, 5, False),
    (24, 640, 6, 7, False), (1024, 512, 4, 4, False), (40, 1024, 4, 5, False), (48, 1280, 3, 4, False),
    (32, 64, 12, 5, False), (60, 100, 4, 6, False),
]


@pytest.mark.parametrize("H,W,K,n,per_label", CASES)
def test_iterations_in_one_call_match(oracle_mod, H, W, K, n, per_label):
    torch = need_cuda()
    from paper_1112_1805_gb300 import binding as B
    from paper_1112_1805_gb300.api import TVSegmenter

    rng = np.random.default_rng(H + W + K)
    img = rng.uniform(0.0, 1.0, (1, H, W)).astype(np.float32)
    cb = np.linspace(0.1, 0.9, K)[:, None]
    lam = float(np.float32(0.08))
    f = torch.tensor(img, device="cuda")
    one, many = TVSegmenter(f, cb, lam, 1.0, per_label), TVSegmenter(f, cb, lam, 1.0, per_label)
    for _ in range(n):
        one.step(1)
    many.step(n - 2)
    many.step(2)
    o = oracle_mod.tv_admm_run(img.astype(np.float64), cb.astype(np.float32).astype(np.float64), lam, 1.0, n, per_label)
    for name in ("u", "w", "bw", "bv", "v"):
        a = one.get(getattr(B, "SEG_" + name.upper())).cpu().numpy()
        b = many.get(getattr(B, "SEG_" + name.upper())).cpu().numpy()
        assert np.abs(a - b).max() <= 1e-4, name
        if name in o:
            assert np.abs(b - np.asarray(o[name]).reshape(b.shape)).max() <= 1e-4, name
    assert int(many.get(B.SEG_ITER)) == n
    one.close()
    many.close()


def test_a_nan_in_the_iterate_stays_one():
    # the closed-form projection must not drop it
    torch = need_cuda()
    from paper_1112_1805_gb300 import binding as B
    from paper_1112_1805_gb300.api import TVSegmenter

    seg = TVSegmenter(torch.rand((64, 64), device="cuda"), np.array([[0.2], [0.5], [0.8]]), 0.05)
    bw = torch.zeros((3, 64, 64), device="cuda")
    bw[1, 5, 7] = float("nan")
    seg.set(B.SEG_BW, bw)
    seg.step(3)
    assert torch.isnan(seg.get(B.SEG_W)).any()
    seg.close()

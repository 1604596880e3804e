"""GPU: TV iterates do not depend on how the iterations are split over calls.  A call
of several iterations runs the row half of all but the last in one kernel, a call
of one runs separate kernels; both have to give the same bits, whichever row
transform the width has (16, 12 or 20 values per thread), with register-FFT and
staged columns, for both group forms and at ragged bands."""

import numpy as np
import pytest

from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,K,per_label", [
    (64, 64, 3, False), (9, 48, 2, False), (8, 80, 8, True), (81, 96, 4, False), (125, 128, 5, True), (45, 192, 4, False),
    (320, 160, 3, True), (512, 128, 4, False), (512, 256, 4, True), (512, 512, 4, False), (300, 320, 2, False),
    (24, 640, 6, False), (1024, 512, 4, False), (40, 1024, 4, False), (48, 1280, 3, False), (32, 64, 12, False),
])
def test_split_calls_give_the_same_bits(H, W, K, per_label):
    torch = need_cuda()
    from paper_1112_1805_gb300 import binding as B
    from paper_1112_1805_gb300.api import TVSegmenter

    g = torch.Generator(device="cuda").manual_seed(H + W + K)
    f = torch.rand((H, W), device="cuda", generator=g)
    cb = np.linspace(0.1, 0.9, K)[:, None]
    ref = None
    for split in ((7,), (1,) * 7, (3, 4), (1, 5, 1), (2, 1, 4)):
        seg = TVSegmenter(f, cb, 0.08, 1.0, per_label)
        for n in split:
            seg.step(n)
        got = [seg.get(x) for x in (B.SEG_U, B.SEG_W, B.SEG_BW, B.SEG_BV, B.SEG_V)]
        seg.close()
        if ref is None:
            ref = got
        for name, a, b in zip(("u", "w", "bw", "bv", "v"), ref, got):
            assert torch.equal(a, b), (split, name, float((a - b).abs().max()))

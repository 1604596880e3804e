"""GPU: the TV state's check for NaN and Inf counts the image at hand only: a
state that refused an image takes the next one."""

import numpy as np
import pytest

from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def test_a_refused_image_does_not_spoil_the_next():
    torch = need_cuda()
    from paper_1112_1805_gb300 import binding as B
    from paper_1112_1805_gb300.api import TVSegmenter

    img = torch.rand((1, 24, 32), device="cuda")
    seg = TVSegmenter(img, np.array([[0.2], [0.8]]), 0.1, 1.0)
    bad = img.clone()
    bad[0, 3, 5] = float("nan")
    with pytest.raises(B.ShearsegError) as e:
        seg.reset(bad)
    assert e.value.code == B.SHF_ERR_NONFINITE
    seg.reset(img)
    seg.step(2)
    assert torch.isfinite(seg.get(B.SEG_U)).all()
    seg.close()

"""GPU: the ADMM of the general path against the oracle's trajectory, at the sizes
that meet each v-step kernel of the rows: heights without register-FFT columns
(odd ones too: a kernel on pairs of rows would leave the last row out) with half
widths of 8, 16 (pairs of rows and single ones), 12, 20 and 32 values per thread.
Bars as in test_gpu_admm.py: max |x - x_oracle| <= 1e-4 for u, w, b_w and b_v,
relative energy error <= 1e-5, labels equal except at top-two gaps below 1e-4."""

import numpy as np
import pytest

from paper_1112_1805_gb300 import synth
from tests.gpu_util import labels_agree, need_cuda

pytestmark = pytest.mark.gpu

CASES = [  # H, W, K, J, C, T
    # odd heights at the half widths whose default is a pair of rows (64, 128)
    (9, 128, 3, 1, 1, 12), (45, 128, 3, 2, 1, 10), (75, 128, 4, 2, 3, 8), (135, 256, 3, 2, 1, 6),
    (225, 256, 2, 3, 1, 5), (27, 256, 9, 2, 1, 8),  # K = 9: the general u/w-step
    # even heights there: pairs of rows
    (50, 128, 3, 2, 1, 10), (90, 256, 4, 2, 1, 6),
    # single rows of 16 values (256, 512) and of 32 (1024)
    (45, 512, 3, 2, 1, 6), (27, 1024, 2, 1, 1, 6), (27, 2048, 2, 1, 1, 5), (18, 2048, 2, 1, 1, 5),
    # 12 and 20 values per thread (L = 24, 96; 40, 320)
    (45, 48, 3, 2, 1, 10), (25, 192, 4, 2, 1, 8), (15, 80, 5, 1, 1, 10), (50, 640, 3, 2, 1, 5),
    # 8 values per thread (L = 8, 32, 768)
    (45, 16, 3, 1, 1, 10), (75, 64, 3, 2, 1, 10), (27, 1536, 2, 1, 1, 5),
]


@pytest.mark.parametrize("H,W,K,J,C,T", CASES)
def test_admm_on_register_rows_at_general_heights(oracle_mod, H, W, K, J, C, T):
    torch = need_cuda()
    from paper_1112_1805_gb300 import binding as B
    from paper_1112_1805_gb300.api import FilterBank, ShearletSegmenter

    rng = np.random.default_rng(H * 5 + W + K)
    cb = rng.uniform(0.1, 0.9, (K, C)) if C == 3 else np.linspace(0.1, 0.9, K)[:, None]
    img, _ = synth.ellipse_image(H, W, cb, rng, n_ellipses=3)
    img = img.astype(np.float32)
    lam = synth.scale_weights(0.1, J).astype(np.float32)
    cb = cb.astype(np.float32)
    fb = FilterBank(H, W, J)
    seg = ShearletSegmenter(fb, torch.tensor(img, device="cuda"), cb, lam.tolist(), 1.0)
    assert seg.plan()["fast"] == 0
    seg.step(T)
    o = oracle_mod.admm_run(img.astype(np.float64), cb.astype(np.float64), J, lam.astype(np.float64), 1.0, T)
    for name in ("u", "w", "bw", "bv"):
        got = seg.get(getattr(B, "SEG_" + name.upper())).cpu().numpy()
        assert np.abs(got - o[name].reshape(got.shape)).max() <= 1e-4, name
    assert abs(seg.energy() - o["energy"]) / abs(o["energy"]) <= 1e-5
    assert labels_agree(seg.labels().cpu().numpy(), o["labels"], o["gap"])
    seg.close()
    fb.close()

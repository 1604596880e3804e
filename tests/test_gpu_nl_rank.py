"""GPU: the candidate ranking of the NL-means graph where FP32 distances cannot
decide the order by themselves: equal patches (an image without noise, a
periodic one), patches that differ in the last bits, values beyond and far below
the range of the FP32 distances, patch weights below it, and the smallest and
largest windows and patches at ragged sizes.  The graph is integer work and must
equal the oracle's."""

import numpy as np
import pytest

from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def _img(kind, H, W, C, seed=5):
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:H, 0:W].astype(np.float64)
    if kind == "flat":
        a = np.where((y - H / 2) ** 2 + (x - W / 3) ** 2 < (H / 4) ** 2, 0.7, 0.3)
    elif kind == "periodic":
        a = 0.5 + 0.2 * np.sin(2 * np.pi * (x + 2 * y) / 8)
    elif kind == "near":
        a = 0.5 + 0.2 * np.sin(2 * np.pi * x / 8) + 1e-7 * rng.standard_normal((H, W))
    else:
        a = rng.standard_normal((H, W)) * {"noise": 1.0, "huge": 1e7, "tiny": 1e-22}[kind]
    return np.stack([a + 0.1 * c * np.roll(a, c, 1) for c in range(C)]).astype(np.float32)


@pytest.mark.parametrize("kind,H,W,C,prm", [
    ("flat", 24, 34, 1, {}), ("periodic", 24, 40, 1, {}), ("near", 33, 40, 1, {}), ("huge", 20, 30, 1, {}),
    ("tiny", 20, 30, 1, {}), ("noise", 33, 66, 3, {"patch": 9}), ("near", 17, 30, 3, {"patch": 1, "window": 3, "neighbours": 1}),
    ("noise", 8, 8, 1, {"neighbours": 8}), ("noise", 25, 36, 1, {"a": 0.1}), ("flat", 12, 70, 3, {"neighbours": 8}),
])
def test_ranking_equals_the_oracle(oracle_mod, kind, H, W, C, prm):
    torch = need_cuda()
    from paper_1112_1805_gb300.api import NLSegmenter

    img = _img(kind, H, W, C)
    cb = np.linspace(0.2, 0.8, 3 * C).reshape(3, C)
    seg = NLSegmenter(torch.tensor(img, device="cuda"), cb, 0.05, 0.2, **prm)
    nbr, deg, _ = seg.graph()
    seg.close()
    onbr, odeg = oracle_mod.nl_graph(img.astype(np.float64), p=prm.get("patch", 5), win=prm.get("window", 15),
                                     a=prm.get("a", 2.0), mt=prm.get("neighbours", 5))
    assert np.array_equal(deg, odeg)
    assert np.array_equal(nbr, onbr)

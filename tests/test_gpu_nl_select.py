"""GPU: the wavefront selection of the NL-means links against the oracle's raster
loop, link for link: images narrower than the window and one row of tiles high,
rows that outnumber the half warps of the CTA (a step takes several turns), ranks
held in more than one piece, counts in memory, and images where nearly every candidate is full or tied."""

import numpy as np
import pytest

from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,flat,prm", [
    (70, 8, False, {}), (8, 90, False, {}), (33, 241, False, {"window": 3}), (64, 66, True, {}),
    (40, 50, True, {"neighbours": 8, "window": 5}), (90, 50, False, {"neighbours": 1, "window": 7}),
    (70, 1000, False, {"patch": 1}),   # 67 rows in a step, 64 half warps
    (500, 200, False, {"window": 3, "neighbours": 4}),
    (1000, 1100, False, {"patch": 1}),  # ranks of 281.6 MB in two pieces of at most 256 MiB
    (40, 1700, False, {"patch": 1}),    # 128 rows in reach: counts not in shared memory
])
def test_links_equal_the_raster_loop(oracle_mod, H, W, flat, prm):
    torch = need_cuda()
    from paper_1112_1805_gb300.api import NLSegmenter

    rng = np.random.default_rng(H + W)
    img = np.full((1, H, W), 0.5, np.float32) if flat else rng.standard_normal((1, H, W)).astype(np.float32)
    seg = NLSegmenter(torch.tensor(img, device="cuda"), np.linspace(0.2, 0.8, 3).reshape(3, 1), 0.05, 0.2, **prm)
    nbr, deg, _ = seg.graph()
    seg.close()
    onbr, odeg = oracle_mod.nl_graph(img.astype(np.float64), p=prm.get("patch", 5), win=prm.get("window", 15),
                                     a=2.0, mt=prm.get("neighbours", 5))
    assert np.array_equal(deg, odeg)
    assert np.array_equal(nbr, onbr)

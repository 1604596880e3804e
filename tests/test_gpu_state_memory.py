"""GPU: a state's buffers come from a pool that banks and states share: states
and banks created and destroyed in any order, on several threads and streams,
give the same results, and the second sweep of an unrolled state (captured) the
same as the first (launched directly) and the third (replayed)."""

import threading

import numpy as np
import pytest

from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def _solve(torch, f, cb, lam, J, n):
    from paper_1112_1805_gb300 import binding as B
    from paper_1112_1805_gb300.api import FilterBank, ShearletSegmenter

    fb = FilterBank(f.shape[0], f.shape[1], J)
    seg = ShearletSegmenter(fb, f, cb, lam)
    seg.step(n)
    u = seg.get(B.SEG_U).clone()
    torch.cuda.synchronize()
    return fb, seg, u


def test_states_and_banks_in_any_order_and_on_threads():
    torch = need_cuda()
    g = torch.Generator(device="cuda").manual_seed(1)
    f = torch.rand((96, 160), device="cuda", generator=g)
    cb, lam = np.array([[0.2], [0.5], [0.8]]), [0.0, 0.01, 0.02]
    fb, seg, ref = _solve(torch, f, cb, lam, 2, 7)
    seg.close()
    fb.close()  # the last user of the pool
    fb, seg, u = _solve(torch, f, cb, lam, 2, 7)
    fb2, seg2, u2 = _solve(torch, f, cb, lam, 2, 7)
    fb.close()  # while another bank and two states live
    seg2.close()
    seg.close()
    fb2.close()
    assert torch.equal(u, ref) and torch.equal(u2, ref)
    got, errors = [], []

    def work():
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(4):
                    b, s, x = _solve(torch, f, cb, lam, 2, 7)
                    got.append(x)
                    s.close()
                    b.close()
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(e)

    threads = [threading.Thread(target=work) for _ in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    torch.cuda.synchronize()
    assert len(got) == 12 and all(torch.equal(x, ref) for x in got)


@pytest.mark.parametrize("H,W", [(64, 128), (30, 50)])
def test_repeated_unrolled_sweeps_give_the_same_bits(H, W):
    torch = need_cuda()
    from paper_1112_1805_gb300 import binding as B
    from paper_1112_1805_gb300.api import FilterBank, ShearletSegmenter

    g = torch.Generator(device="cuda").manual_seed(2)
    f = torch.rand((H, W), device="cuda", generator=g)
    fb = FilterBank(H, W, 2)
    seg = ShearletSegmenter(fb, f, np.array([[0.2], [0.5], [0.8]]), [0.0, 0.01, 0.02])
    gw = torch.randn((3, H, W), device="cuda", generator=g)
    torch.cuda.synchronize()
    runs = []
    for T, ck in ((6, 3), (6, 3), (6, 3), (4, 4), (6, 3), (6, 3)):
        B.seg_admm_unrolled_fwd(seg.handle, T, ck)
        w = seg.get(B.SEG_W).clone()
        dc, dl = B.seg_admm_unrolled_bwd(seg.handle, gw.data_ptr(), 3, 1, 2, 0)
        runs.append((T, w, np.array(dc), np.array(dl)))
    first = runs[0]
    for T, w, dc, dl in runs[1:]:
        if T == 6:
            assert torch.equal(w, first[1]) and np.array_equal(dc, first[2]) and np.array_equal(dl, first[3])
    seg.close()
    fb.close()

"""GPU parity of the transform on each of its routes, at the sizes where they
meet: whole planes in shared memory (and just past it, by size and by number of
planes), register-FFT columns with and without register-FFT rows, staged columns
with register-FFT rows, and staged kernels in several waves; single and many
channels.  Bounds as in test_gpu_transform.py: 2e-5 of the largest value."""

import numpy as np
import pytest

from tests.gpu_util import need_cuda, rel_max_err

pytestmark = pytest.mark.gpu

SIZES = [
    (9, 8, 1, 1), (8, 250, 1, 3), (36, 216, 2, 2),   # whole planes, up to 5000 values for the synthesis
    (90, 120, 3, 2), (108, 250, 3, 1),               # ... past that; the largest plane
    (16, 16, 1, 128),                                # more planes than whole-plane CTAs are used for
    (128, 144, 3, 5), (256, 162, 3, 2),              # register-FFT columns, staged rows (L = 72, 81)
    (64, 1536, 2, 2),                                # L = 768: staged rows at a register-FFT width
    (135, 256, 2, 3), (250, 640, 3, 2),              # staged columns, register-FFT rows
    (270, 600, 3, 2), (45, 2000, 2, 1),              # staged both ways
]


@pytest.mark.parametrize("H,W,J,nch", SIZES)
def test_routes_match_the_oracle(oracle_mod, H, W, J, nch):
    torch = need_cuda()
    from paper_1112_1805_gb300.api import FilterBank

    rng = np.random.default_rng(H * 13 + W)
    u = rng.standard_normal((nch, H, W)).astype(np.float32)
    fb = FilterBank(H, W, J)
    got = fb.analyze(torch.tensor(u, device="cuda"))
    ref = oracle_mod.analyze(u.astype(np.float64), J)
    assert rel_max_err(got.cpu().numpy(), ref) < 2e-5
    c = rng.standard_normal((nch, fb.eta, H, W)).astype(np.float32)
    back = fb.synthesize(torch.tensor(c, device="cuda")).cpu().numpy()
    assert rel_max_err(back, oracle_mod.synthesize(c.astype(np.float64), J)) < 2e-5
    fb.close()


@pytest.mark.parametrize("H,W,J,nch", [(1024, 1000, 4, 2), (1080, 1024, 4, 2), (1620, 1800, 4, 1), (2048, 1024, 4, 2)])
def test_several_waves_are_a_parseval_frame(H, W, J, nch):
    # more spectra than one wave holds: S^T S = I, |S u| = |u| and <S u, c> = <u, S^T c>
    torch = need_cuda()
    from paper_1112_1805_gb300.api import FilterBank

    g = torch.Generator(device="cuda").manual_seed(H + W)
    u = torch.randn((nch, H, W), device="cuda", generator=g)
    fb = FilterBank(H, W, J)
    c = fb.analyze(u)
    r = fb.synthesize(c)
    assert float((r - u).abs().max()) < 2e-5 * float(u.abs().max())
    assert abs(float(c.double().norm() / u.double().norm()) - 1) < 1e-5
    d = torch.randn(c.shape, device="cuda", generator=g)
    lhs = float((c.double() * d.double()).sum())
    rhs = float((u.double() * fb.synthesize(d).double()).sum())
    # single values are off by 1e-6 of their norms at most
    assert abs(lhs - rhs) < 1e-6 * float(c.double().norm()) * float(d.double().norm())
    fb.close()


def test_calls_on_two_streams_and_under_capture_agree():
    torch = need_cuda()
    from paper_1112_1805_gb300.api import FilterBank

    for H, W, J in ((64, 64, 2), (128, 128, 3), (90, 250, 3)):
        fb = FilterBank(H, W, J)
        u = torch.randn((3, H, W), device="cuda")
        c = fb.analyze(u)
        r = fb.synthesize(c)
        torch.cuda.synchronize()
        outs = []
        for _ in range(2):
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(5):
                    a = fb.analyze(u)
                    b = fb.synthesize(a)
            outs.append((a, b))
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            a = fb.analyze(u)
            b = fb.synthesize(a)
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        for x, y in outs + [(a, b)]:
            assert torch.equal(x, c) and torch.equal(y, r)
        del graph
        fb.close()

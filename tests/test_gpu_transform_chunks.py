"""GPU: the transforms on register-FFT columns with tiles of 8 columns (heights up to
1024) when their spectra take more than one wave of 1024 MiB, by filters (125 planes
of 8.5 MB) and by channels (three of 61 planes): buffers used again from wave to
wave and from chunk to chunk, partial sums per channel.

Chunks of channels run what single channels run: the same bits.  Waves: S^T S = I
to 2e-5 of the largest value and |S u| = |u| to 1e-5 as in
test_gpu_transform_routes.py, and the coefficients of filters in both waves against
FP64 FFTs with the stored filters to 2e-5 of the largest value."""

import pytest

from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def test_channel_chunks_repeat_single_channels():
    torch = need_cuda()
    from paper_1112_1805_gb300.api import FilterBank

    g = torch.Generator(device="cuda").manual_seed(3)
    H, W, J = 1024, 2048, 4
    u = torch.randn((3, H, W), device="cuda", generator=g)
    fb = FilterBank(H, W, J)
    c = fb.analyze(u)
    r = fb.synthesize(c)
    assert float((r - u).abs().max()) < 2e-5 * float(u.abs().max())
    for k in range(3):
        one = fb.analyze(u[k : k + 1])
        assert torch.equal(one[0], c[k])
        assert torch.equal(fb.synthesize(c[k : k + 1])[0], r[k])
        del one
    fb.close()


def test_filter_waves_match_fp64():
    torch = need_cuda()
    from paper_1112_1805_gb300 import binding as B
    from paper_1112_1805_gb300.api import FilterBank

    g = torch.Generator(device="cuda").manual_seed(4)
    H, W, J = 1024, 2048, 5
    u = torch.randn((1, H, W), device="cuda", generator=g)
    fb = FilterBank(H, W, J)
    bank = torch.empty((fb.eta, H, W // 2 + 1), device="cuda")
    B.shfilters_copy(fb.handle, bank.data_ptr(), torch.cuda.current_stream().cuda_stream)
    c = fb.analyze(u)
    spec = torch.fft.rfft2(u[0].double())
    for f in (0, 1, 40, 61, 62, 63, 64, 100, 124):
        ref = torch.fft.irfft2(spec * bank[f].double(), s=(H, W))
        assert float((c[0, f] - ref).abs().max()) < 2e-5 * float(ref.abs().max()), f
    assert abs(float(c.double().norm() / u.double().norm()) - 1) < 1e-5
    assert float((fb.synthesize(c) - u).abs().max()) < 2e-5 * float(u.abs().max())
    fb.close()

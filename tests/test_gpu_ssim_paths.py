"""The SSIM passes fetch four samples at a time where rows start on 16-byte boundaries, one at a time elsewhere:
the same planes at such an address and one float beside it must give the same results.  Tolerances: 22 roundings
of 2^-24 per filtered moment, times 1 / (variance + c2) ~ 10 for these noise images, against the largest
gradient; the sums average those errors."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _planes(gen, v, h, w, shift):
    n = v * 3 * h * w
    buf = torch.empty(n + 4, device="cuda")
    t = buf[shift:shift + n].view(v, 3, h, w)
    t.copy_(torch.rand(v, 3, h, w, generator=gen).cuda())
    return t


@pytest.mark.parametrize("h,w", [(1, 4), (5, 8), (11, 28), (32, 32), (33, 36), (64, 100), (31, 132)])
@pytest.mark.parametrize("refine", [False, True])
def test_aligned_and_unaligned_planes_agree(h, w, refine):
    from paper_2605_10760_gb300 import raster as R
    v, got = 2, []
    for shift in (0, 1):
        gen = torch.Generator().manual_seed(100 * h + w)
        x, y = _planes(gen, v, h, w, shift), _planes(gen, v, h, w, shift)
        if refine:
            expo = torch.tensor([[0.1, -0.02], [-0.05, 0.03]], device="cuda")
            loss, d_rgb, _, d_expo = R.loss_refine(x, y, expo, w_depth=0.0)
            torch.testing.assert_close(d_expo, got[0][2] if got else d_expo, rtol=1e-4, atol=1e-6)
        else:
            loss, d_rgb = R.loss_l1_ssim(x, y, 0.8, 0.2)[:2]
            d_expo = None
        got.append((loss.item(), d_rgb.clone(), d_expo))
    assert (got[0][1] - got[1][1]).abs().max() <= 2e-5 * got[0][1].abs().max()
    assert abs(got[0][0] - got[1][0]) <= 1e-6 * abs(got[0][0])


@pytest.mark.parametrize("h,w", [(1, 3), (2, 2), (5, 7), (64, 100)])
def test_depth_term_agrees_at_both_alignments(h, w):
    """Elementwise gradients are the same bits; the loss is a sum of the same terms in FP64 or better."""
    from paper_2605_10760_gb300 import raster as R
    v, got = 2, []
    for shift in (0, 1):
        gen = torch.Generator().manual_seed(h * w)
        x, y = (torch.rand(v, 3, h, w, generator=gen).cuda() for _ in range(2))
        maps = []
        for _ in range(3):
            buf = torch.empty(v * h * w + 4, device="cuda")
            maps.append(buf[shift:shift + v * h * w].view(v, h, w))
            maps[-1].copy_(torch.rand(v, h, w, generator=gen).cuda())
        loss, _, d_depth, _ = R.loss_refine(x, y, torch.zeros(v, 2, device="cuda"), maps[0], maps[1], 1.0, 0.0, 0.25,
                                            d_depth=maps[2])
        got.append((loss.item(), d_depth.clone()))
        want = torch.sign(maps[0] - maps[1]) * torch.tensor(0.25 / (v * h * w), dtype=torch.float64).float().cuda()
        assert torch.equal(d_depth, want)
    assert abs(got[0][0] - got[1][0]) <= 1e-9 * got[0][0] and torch.equal(got[0][1], got[1][1])

"""The SSIM passes walk strips of 32 columns down segments of 32-row steps, whose length depends on the number of
planes: one and the same plane alone, and repeated often enough that its strips become one long segment, must give
the same gradients.  Tolerance: both ways run the same operations per pixel, so only the 1 / (3 V W H) scale, a
power of two apart, differs: one rounding, 2^-22 with the L1 term's."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,w", [(31, 40), (32, 32), (33, 36), (65, 29), (101, 64), (200, 37)])
@pytest.mark.parametrize("refine", [False, True])
def test_segments_agree(h, w, refine):
    from paper_2605_10760_gb300 import raster as R
    gen = torch.Generator().manual_seed(h * w)
    x, y = (torch.rand(1, 3, h, w, generator=gen).cuda() for _ in range(2))
    got = []
    for v in (1, 1024):
        xs, ys = x.expand(v, -1, -1, -1).contiguous(), y.expand(v, -1, -1, -1).contiguous()
        if refine:
            expo = torch.tensor([[0.1, -0.02]], device="cuda").expand(v, -1).contiguous()
            loss, d_rgb, _, _ = R.loss_refine(xs, ys, expo, w_depth=0.0)
        else:
            loss, d_rgb = R.loss_l1_ssim(xs, ys, 0.8, 0.2)[:2]
        got.append((loss.item(), v * d_rgb[0], v * d_rgb[-1]))
    scale = got[0][1].abs().max()
    for d in got[1][1:]:
        assert (d - got[0][1]).abs().max() <= 2.0 ** -22 * scale * 4
    assert abs(got[1][0] - got[0][0]) <= 1e-9 * abs(got[0][0])

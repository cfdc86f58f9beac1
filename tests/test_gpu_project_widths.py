"""A few chunks are projected by wide blocks, many by narrow ones: one view on its own and the same view repeated until
its chunks are too many for the wide blocks must give the same images, bit for bit, and the same gradients up to the
order of FP32 additions (up to 1000 pose terms or 320 views, n 2^-24 = 6e-5 of the terms' magnitudes, with a sum a
third of them: 2e-4 of the largest)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 63, 256, 257, 1000])
def test_wide_and_narrow_blocks_agree(n):
    from paper_2605_10760_gb300 import raster as R, scenes as S
    g = R.Gaussians.from_scene(S.random_cloud(n, seed=n))
    cam = S.Camera(np.eye(3, dtype=np.float32), np.array([0, 0, 4], np.float32), 60.0, 60.0, 32.0, 24.0, 64, 48)
    chunks = -(-n // 256)
    got = []
    for v in (1, -(-320 // chunks)):
        pb = R.Problem([0] * v, [n] * v, n, 64, 48, cameras=R.cameras_tensor([cam] * v))
        img = pb.forward_checked(g)
        up = torch.linspace(-1, 1, 3 * 48 * 64, device="cuda").view(1, 3, 48, 64).expand(v, -1, -1, -1).contiguous()
        grads = pb.render_bwd(g, img, up)
        got.append(([img[k][0].clone() for k in ("rgb", "depth", "alpha", "last_idx")],
                    [getattr(grads, k) / v for k in ("means", "log_scales", "quats", "opacities", "colors")],
                    pb.pose_grad()))
    assert (got[0][0][2] > 0).any()
    for a, b in zip(got[0][0], got[1][0]):
        assert torch.equal(a, b)
    for a, b in zip(got[0][1] + [got[0][2][0]], got[1][1] + [got[1][2][-1]]):
        assert (a - b).abs().max() <= 2e-4 * a.abs().max() + 1e-12

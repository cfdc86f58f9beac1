"""A sum of |difference| with an infinite term is infinite (a depth map marks pixels without a return so), whether the
loss stands alone, inside the compositing kernel or in the refinement, at both widths of access."""
import numpy as np
import pytest

from helpers import gpu_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2605_10760_gb300 import scenes as S  # noqa: E402


@pytest.mark.parametrize("value,want", [(np.inf, np.inf), (-np.inf, np.inf), (np.nan, np.nan)])
@pytest.mark.parametrize("w,h", [(64, 48), (37, 21)])
def test_infinite_depth_target(w, h, value, want):
    from paper_2605_10760_gb300 import raster as R
    sc = S.random_cloud(300, seed=4)
    wl = S.Workload("t", sc, np.array([0, 300], np.int64), [S.identity_camera(w, h, 60, 60)], np.zeros(1, np.int32), w, h)
    pb, g = gpu_problem(wl)
    img = pb.forward_checked(g)
    rgb_t = torch.rand(1, 3, h, w, device="cuda")
    depth_t = torch.rand(1, h, w, device="cuda")
    depth_t[0, h // 2, ::5] = float(value)
    losses = [R.loss_l1(img["rgb"], rgb_t, img["depth"], depth_t, 1.0, 0.25)[0],
              pb.render_fwd_l1(img, rgb_t, depth_t, 1.0, 0.25)[1],
              R.loss_refine(img["rgb"], rgb_t, torch.zeros(1, 2, device="cuda"), img["depth"], depth_t)[0]]
    for loss in losses:
        np.testing.assert_equal(loss.item(), want)

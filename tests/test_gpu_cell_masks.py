"""The compositing kernels' per-cell skips (a quarter warp's 4 x 4 pixels) never change a decision: round to
needle-shaped footprints at every orientation, opacities below and above alpha_min, every tile shape and
staged batch size, and alpha_min = 0, where no cut-off exists and an opacity of 0 blends too.

Values are compared with the 64-bit oracle for the moderate footprints only: the FP32 sigma of the
decision chain is within 6 u M of the exact quadratic (u = 2^-24, M the magnitude of its terms), and
conic entries of 1e3 at offsets of 50 pixels make M about 1e6."""
import numpy as np
import pytest

from helpers import TOL_GRAD, TOL_IMAGE, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2605_10760_gb300 import scenes as S  # noqa: E402
from test_gpu_parity import run_gpu, run_oracle  # noqa: E402


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_10760_gb300 import raster
    raster.L.load()
    return raster


def ellipses(max_ratio, n=1200, seed=3, W=203, H=149):
    rng = np.random.default_rng(seed)
    sc = S.random_cloud(n, seed=seed)
    sc.means[:, 0] = rng.uniform(-1.6, 1.6, n)
    sc.means[:, 1] = rng.uniform(-1.2, 1.2, n)
    sc.means[:, 2] = rng.uniform(1.5, 4.0, n)
    long_axis = rng.uniform(-4.5, -1.6, n)
    ratio = np.exp(rng.uniform(0.0, np.log(max_ratio), n))
    sc.log_scales[:] = np.stack([long_axis, long_axis - np.log(ratio), long_axis - np.log(ratio)], 1)
    sc.opacities[:] = np.where(rng.random(n) < 0.1, rng.choice([0.0, 1e-4, 0.0039, 0.004], n), rng.uniform(0.02, 0.999, n))
    return S.Workload("ellipses", sc, np.array([0, n], np.int64), [S.identity_camera(W, H, 180, 180, W / 2, H / 2)],
                      np.zeros(1, np.int32), W, H)


@pytest.mark.parametrize("alpha_min", [1.0 / 255.0, 0.0])
@pytest.mark.parametrize("tw,th,nb", [(16, 16, 0), (16, 16, 64), (16, 16, 128), (16, 8, 64), (32, 16, 128), (32, 16, 256)])
@pytest.mark.parametrize("max_ratio", [30.0, 3000.0])
def test_cells_keep_decisions_exact(R, max_ratio, tw, th, nb, alpha_min):
    wl = ellipses(max_ratio)
    p = R.default_params(tile_w=tw, tile_h=th, batch_records=nb, alpha_min=alpha_min, dilation=0.3 if max_ratio < 100 else 1e-3)
    gpu = run_gpu(R, wl, params=p, alpha_w=0.3)
    assert gpu["rc"] == 0 and gpu["rc_end"] == 0
    orc = run_oracle(wl, params=p, up=gpu["up"])
    np.testing.assert_array_equal(gpu["img"]["last_idx"], orc["fwd"]["last"])
    assert gpu["stats"]["fwd_pairs"] == orc["fwd"]["pairs"]
    if max_ratio < 100:
        for k in ("rgb", "depth", "alpha", "final_T"):
            assert np.abs(gpu["img"][k].astype(np.float64) - orc["fwd"][k]).max() <= TOL_IMAGE, k
        for k in ("means", "log_scales", "quats", "opacities", "colors"):
            assert rel_l2(gpu["grads"][k], orc["bwd"][k]) <= TOL_GRAD, k

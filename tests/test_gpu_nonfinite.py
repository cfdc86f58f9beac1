"""Infinities and NaN stay where they are blended: a colour, a far depth or an upstream gradient that is not finite
reaches the pixels that blend its Gaussian and the Gaussians that its pixel blends, and no others, whatever else
shares their cell of 4 x 4 pixels, their staged batch or their tile.

Gradients are sums of FP32 atomics in any order: n terms differ by less than n 2^-24 of their magnitudes' sum.  The
grid's Gaussians collect fewer than 16 quarter-warp sums each (2^-20; not the quaternions' gradient, which is nothing
but the rounding of terms that cancel for its round footprints); the crowd's are held to 1e-4 of the tensor's largest
entry."""
import numpy as np
import pytest

from helpers import gpu_problem, upstream

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2605_10760_gb300 import scenes as S  # noqa: E402

FIELDS = ("means", "log_scales", "quats", "opacities", "colors")
BAD = (np.nan, np.inf, -np.inf, 3e38)
SHAPES = [(16, 16, 0), (16, 16, 64), (16, 16, 128), (16, 8, 64), (32, 16, 256)]


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_10760_gb300 import raster
    raster.L.load()
    return raster


def crowd(n=1500, W=203, H=149, seed=11):
    """Overlapping footprints, a third of them too transparent to be blended anywhere."""
    rng = np.random.default_rng(seed)
    sc = S.random_cloud(n, seed=seed)
    sc.log_scales[:] = rng.uniform(-5.0, -2.5, (n, 3))
    clear = rng.random(n) < 0.33
    sc.opacities[:] = np.where(clear, rng.choice([0.0, 1e-4, 0.0038], n), rng.uniform(0.05, 0.95, n))
    cam = S.identity_camera(W, H, 110.0, 110.0, W / 2, H / 2)
    return S.Workload("crowd", sc, np.array([0, n], np.int64), [cam], np.zeros(1, np.int32), W, H), np.nonzero(clear)[0]


def grid(W=96, H=64, step=5):
    """Small footprints (1.8 pixels, the dilation's own) one beside another: no pixel blends two of them."""
    x, y = np.meshgrid(np.arange(3, W, step), np.arange(3, H, step))
    n = x.size
    sc = S.random_cloud(n, seed=2)
    sc.means[:] = np.stack([(x.ravel() + 0.5 - W / 2) / 50, (y.ravel() + 0.5 - H / 2) / 50, np.full(n, 2.0)], 1)
    sc.log_scales[:] = -9.0
    sc.opacities[:] = 0.9
    cam = S.identity_camera(W, H, 100.0, 100.0, W / 2, H / 2)
    return S.Workload("grid", sc, np.array([0, n], np.int64), [cam], np.zeros(1, np.int32), W, H)


def forward(R, wl, shape, **kw):
    tw, th, nb = shape
    pb, g = gpu_problem(wl, params=R.default_params(tile_w=tw, tile_h=th, batch_records=nb, **kw))
    return pb, g, pb.forward_checked(g)


def backward(pb, g, img, up):
    gr = pb.render_bwd(g, img, *[None if u is None else torch.as_tensor(u).cuda() for u in up])
    pose = pb.pose_grad()
    assert pb.check_status()[0] == 0
    return {k: getattr(gr, k).cpu().numpy() for k in FIELDS} | {"pose": pose.cpu().numpy()}


def assert_images(a, b):
    for k in b:
        assert np.array_equal(a[k].cpu().numpy().view(np.uint32), b[k].cpu().numpy().view(np.uint32)), k


@pytest.mark.parametrize("alpha_min", [1.0 / 255.0, 1e-37])    # the second: cut-offs beyond the short exponential's range
@pytest.mark.parametrize("shape", SHAPES)
def test_gaussians_that_nothing_blends_reach_nothing(R, shape, alpha_min):
    wl, clear = crowd()
    if alpha_min < 1e-30:
        wl.scene.opacities[clear] = 0.0
    up = upstream(wl, 1, alpha_w=0.3)
    wl.scene.colors[clear] = 0.0
    pb, g, want = forward(R, wl, shape, alpha_min=alpha_min)
    grads = backward(pb, g, want, up)
    wl.scene.colors[clear] = np.resize(BAD, (len(clear), 3)).astype(np.float32)
    pb, g, got = forward(R, wl, shape, alpha_min=alpha_min)
    assert_images(got, want)
    for k, x in backward(pb, g, got, up).items():
        assert np.isfinite(x).all(), k
        assert np.abs(x - grads[k]).max() <= 1e-4 * np.abs(grads[k]).max(), k


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("shape", SHAPES)
def test_a_colour_stays_in_the_pixels_that_blend_it(R, shape, bad):
    wl, clear = crowd()
    seen = np.setdiff1d(np.arange(wl.scene.n), clear)[::7]
    colors = wl.scene.colors.copy()
    wl.scene.colors[:] = 0.0
    wl.scene.colors[seen] = 1.0
    blends = forward(R, wl, shape)[2]["rgb"].cpu().numpy() > 0
    wl.scene.colors[:] = colors
    wl.scene.colors[seen] = 0.0
    want = {k: v.cpu().numpy() for k, v in forward(R, wl, shape)[2].items()}
    wl.scene.colors[seen] = np.array([bad, 0.5, bad], np.float32)
    got = {k: v.cpu().numpy() for k, v in forward(R, wl, shape)[2].items()}
    assert 0 < blends.sum() < blends.size
    for c in (0, 2):
        np.testing.assert_array_equal(got["rgb"][:, c][~blends[:, c]], want["rgb"][:, c][~blends[:, c]])
        if not np.isfinite(bad):
            assert not np.isfinite(got["rgb"][:, c][blends[:, c]]).any()
    assert np.isfinite(got["rgb"][:, 1]).all()
    for k in ("depth", "alpha", "final_T", "last_idx"):
        np.testing.assert_array_equal(got[k], want[k])


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("shape", SHAPES)
def test_gradients_beside_a_colour_and_an_upstream_value(R, shape, bad):
    wl = grid()
    up = [u.copy() for u in upstream(wl, 1, alpha_w=0.3)]
    pb, g, want = forward(R, wl, shape)
    grads = backward(pb, g, want, up)

    def check(x, others):
        for k in FIELDS:
            d = np.abs(x[k] - grads[k])[others]
            assert np.isfinite(x[k][others]).all(), k
            assert k == "quats" or d.max() <= 2.0 ** -20 * np.abs(grads[k]).max(), k

    # every third Gaussian's colour
    other = np.arange(wl.scene.n) % 3 != 1
    colors = wl.scene.colors.copy()
    wl.scene.colors[~other, 0] = bad
    pb, g, img = forward(R, wl, shape)
    check(backward(pb, g, img, up), other)
    wl.scene.colors[:] = colors
    # the upstream values of some Gaussians' centre pixels, one array at a time
    last = want["last_idx"][0].cpu().numpy()
    for a, pick in enumerate((np.s_[0, 1, 8::10, 8::10], np.s_[0, 8::10, 8::10], np.s_[0, 8::10, 8::10])):
        hit = np.zeros_like(last, bool)
        hit[8::10, 8::10] = True
        assert (last[hit] > 0).all()
        yy, xx = np.nonzero(hit)
        owner = ((yy - 3) // 5) * len(range(3, wl.width, 5)) + (xx - 3) // 5
        other = np.ones(wl.scene.n, bool)
        other[owner] = False
        bent = [u.copy() for u in up]
        bent[a][pick] = bad
        pb, g, img = forward(R, wl, shape)
        check(backward(pb, g, img, bent), other)


@pytest.mark.parametrize("bad", BAD[:2])
@pytest.mark.parametrize("shape", SHAPES)
def test_gradients_of_gaussians_that_no_spoilt_pixel_blends(R, shape, bad):
    """Lists of several batches: a pixel that has met a bad colour keeps its spoilt sums to the entries it blends, in the
    batches in front of that colour's too."""
    wl, clear = crowd(n=9000)
    up = upstream(wl, 1, alpha_w=0.3)
    seen = np.setdiff1d(np.arange(wl.scene.n), clear)[::1000]
    colors = wl.scene.colors.copy()
    wl.scene.colors[:] = 0.0
    wl.scene.colors[seen] = 1.0
    spoilt = (forward(R, wl, shape)[2]["rgb"] > 0).any(1, keepdim=True).float().expand(1, 3, -1, -1).contiguous()
    wl.scene.colors[:] = colors
    wl.scene.colors[seen] = 0.0
    pb, g, img = forward(R, wl, shape)
    assert int(pb.workspace()["tile_ranges"].diff(dim=1).max()) > 600
    others = backward(pb, g, img, (spoilt, None, None))["colors"][:, 1] == 0
    others[clear] = True
    assert 0.05 < others.mean() < 0.95 and 0.005 < float(spoilt.mean()) < 0.6
    grads = backward(pb, g, img, up)
    wl.scene.colors[seen] = np.float32(bad)
    pb, g, img = forward(R, wl, shape)
    got = backward(pb, g, img, up)
    for k in FIELDS:
        assert np.isfinite(got[k][others]).all(), k
        assert np.abs(got[k] - grads[k])[others].max() <= 1e-4 * np.abs(grads[k]).max(), k

"""Binning: both algorithms against numpy's sort by (depth bits, pair index), at the list lengths where
the tile-first one changes its method (registers of a warp, shared memory of a CTA, merged runs) and at
the tile counts and batch shapes that the radix one splits into digits."""
import numpy as np
import pytest

from helpers import gpu_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2605_10760_gb300 import scenes as S  # noqa: E402


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_10760_gb300 import raster
    raster.L.load()
    return raster


def workload(n, W, H, views=1, ties=False, seed=5):
    sc = S.random_cloud(n, seed=seed)
    if ties:   # many equal depths: the pair index decides
        sc.means[:, 2] = np.round(sc.means[:, 2] * 8) / 8
    cams = [S.look_at((0.02 * v, 0.0, 0.0), (0.02 * v, 1e-3, 4.0), W, H, 0.9 * W, 0.9 * W, W / 2, H / 2) for v in range(views)]
    return S.Workload("bin", sc, np.array([0, n], np.int64), cams, np.zeros(views, np.int32), W, H)


def binned(R, wl, mode, cap=None):
    pb, g = gpu_problem(wl, params=R.default_params(sort_mode=mode), key_capacity=cap)
    pb.project(g)
    counts = pb.workspace()["tiles_touched"].clone()
    pb.bin_sort()
    rc, req = pb.check_status()
    ws = pb.workspace()
    K = int(ws["num_keys"][0].item())
    out = dict(pb=pb, g=g, rc=rc, req=req, K=K, counts=counts.cpu().numpy().view(np.uint32).astype(np.int64))
    if rc == 0:
        out["keys"] = ws["sorted_keys"][:K].cpu().numpy().view(np.uint64)
        out["vals"] = ws["sorted_vals"][:K].cpu().numpy().view(np.uint32)
        out["ranges"] = ws["tile_ranges"].cpu().numpy().view(np.uint32).astype(np.int64)
        out["touched"] = ws["tiles_touched"].cpu().numpy().view(np.uint32).astype(np.int64)
        out["proj"] = ws["proj"].cpu().numpy()
        out["claims"] = int(ws["claim_count"].sum().item())
    assert pb.check_guards() == (0, -1)
    return out


def expected(wl, got):
    """Sorted keys and values from the projection records: rectangles, then numpy's lexsort."""
    vis = np.nonzero(got["counts"])[0]
    p = got["proj"][vis]
    tx, ty = -(-wl.width // 16), -(-wl.height // 16)
    f32 = np.float32
    lo = lambda m, n: np.clip(np.floor((m - p[:, 7]) / f32(16)), 0, n).astype(np.int64)
    hi = lambda m, n: np.clip(np.floor((m + p[:, 7]) / f32(16)) + 1, 0, n).astype(np.int64)
    x0, x1, y0, y1 = lo(p[:, 0], tx), hi(p[:, 0], tx), lo(p[:, 1], ty), hi(p[:, 1], ty)
    nx, cnt = x1 - x0, (x1 - x0) * (y1 - y0)
    np.testing.assert_array_equal(cnt, got["counts"][vis])
    e = np.repeat(np.arange(len(vis)), cnt)
    k = np.arange(cnt.sum()) - np.repeat(np.cumsum(cnt) - cnt, cnt)
    tile = (vis[e] // wl.scene.n) * tx * ty + (y0[e] + k // nx[e]) * tx + x0[e] + k % nx[e]
    z = p[:, 6].view(np.uint32).astype(np.uint64)[e]
    order = np.lexsort((vis[e], z, tile))
    return (tile.astype(np.uint64)[order] << np.uint64(32)) | z[order], vis[e][order], tile[order]


def check(R, wl, mode):
    got = binned(R, wl, mode)
    assert got["rc"] == 0
    keys, vals, tile = expected(wl, got)
    assert got["K"] == len(keys)
    np.testing.assert_array_equal(got["keys"], keys)
    np.testing.assert_array_equal(got["vals"], vals)
    G = len(got["ranges"])
    start, end = np.searchsorted(tile, np.arange(G), "left"), np.searchsorted(tile, np.arange(G), "right")
    np.testing.assert_array_equal(got["ranges"], np.stack([np.where(end > start, start, 0), np.where(end > start, end, 0)], 1))
    assert got["claims"] == G
    want = np.cumsum(got["counts"]) if mode == 1 else got["counts"]
    np.testing.assert_array_equal(got["touched"], want)
    return got


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2047, 2048,
                               2049, 4097, 8191, 8192, 8193, 16385, 24577])
def test_tile_first_list_lengths(R, n, ties):
    """One 16x16 tile, so the list holds every visible Gaussian (about n)."""
    check(R, workload(n, 16, 16, ties=ties), 0)


@pytest.mark.parametrize("n", [257, 1024, 1025, 2048, 2049, 4096, 4097, 9000])
def test_tile_first_long_lists_among_many_tiles(R, n):
    """More tiles than SMs: 256-thread CTAs, whose runs hold 2048 words; a pile of about n Gaussians in the
    central tiles beside short lists."""
    wl = workload(n, 320, 240)
    wl.scene.means[: 9 * n // 10, :2] *= 0.02
    check(R, wl, 0)


@pytest.mark.parametrize("n,W,H,views", [(16_385, 16, 16, 1), (33_000, 32, 16, 1), (60_000, 33, 17, 1), (150_000, 40, 40, 1),
                                         (33_000, 31, 9, 40), (17_000, 16, 16, 300), (1025, 640, 480, 1), (40_000, 160, 120, 1),
                                         (3_001, 48, 32, 1024)])
def test_binning_modes_agree_with_numpy(R, n, W, H, views):
    """Shapes whose pairs per tile send the default mode through the radix binning (0 to 11 tile bits, one
    view to hundreds), and some that do not, each in both modes."""
    wl = workload(n, W, H, views, ties=views > 1)
    one, zero = check(R, wl, 1), check(R, wl, 0)
    imgs = [o["pb"].render_fwd() for o in (one, zero)]
    for k in imgs[0]:
        assert torch.equal(imgs[0][k], imgs[1][k]), k


@pytest.mark.parametrize("mode", [1, 0])
def test_capacity_in_both_binnings(R, mode):
    """Too few keys: the number needed is reported, nothing is written beyond, and the next call with room
    is complete (one tile, so the default mode takes the radix binning)."""
    wl = workload(17_000, 16, 16)
    small = binned(R, wl, mode, cap=1000)
    assert small["rc"] == R.L.GS_ERR_CAPACITY and small["req"] == small["counts"].sum()
    pb = small["pb"]
    pb.set_capacity(int(small["req"]))
    pb.project(small["g"])
    pb.bin_sort()
    assert pb.check_status()[0] == 0 and pb.check_guards() == (0, -1)
    check(R, wl, mode)

"""Views whose Gaussians pile up in a few tiles: lists long enough that the sorting CTAs share them, at the lengths
where the number of runs and of merge levels changes, of several lengths at once and beside short lists, against
numpy's sort by (depth bits, pair index); and the time that a pile takes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2605_10760_gb300 import scenes as S  # noqa: E402
from helpers import gpu_problem  # noqa: E402
from test_gpu_binning import R, check  # noqa: E402,F401


def piles(lengths, W, H, spread=700, seed=9):
    """lengths[k] Gaussians of 2 pixels' radius around the middle of a tile of their own, `spread` ones anywhere; a
    tenth of the depths equal another's."""
    rng = np.random.default_rng(seed)
    n = int(np.sum(lengths)) + spread
    tx, ty = W // 16, H // 16
    tile = rng.permutation(tx * ty)[:len(lengths)]
    owner = np.repeat(tile, lengths)
    px = np.concatenate([owner % tx * 16 + 8 + rng.uniform(-4, 4, len(owner)), rng.uniform(0, W, spread)])
    py = np.concatenate([owner // tx * 16 + 8 + rng.uniform(-4, 4, len(owner)), rng.uniform(0, H, spread)])
    z = rng.uniform(2, 4, n).astype(np.float32)
    z[rng.integers(0, n, n // 10)] = z[rng.integers(0, n, n // 10)]
    sc = S.random_cloud(n, seed=seed)
    sc.means[:] = np.stack([(px - W / 2) * z / 200, (py - H / 2) * z / 200, z], 1)
    sc.log_scales[:] = -9.0
    p = rng.permutation(n)      # a pile's Gaussians are spread over the pairs
    sc.means[:] = sc.means[p]
    cam = S.identity_camera(W, H, 200.0, 200.0, W / 2, H / 2)
    return S.Workload("piles", sc, np.array([0, n], np.int64), [cam], np.zeros(1, np.int32), W, H)


# more tiles than SMs (CTAs of 256 threads, runs of 2048 words), then fewer (1024 threads, 8192 words)
@pytest.mark.parametrize("W,H", [(320, 240), (96, 64)])
@pytest.mark.parametrize("lengths", [(2000,), (4090, 4100, 8200), (16380, 16390, 9000), (18432, 18433, 20480, 20481), (32768, 32769, 4000, 300),
                                     (140_000, 35_000, 17_000, 16_400, 2_500), (600_000, 30_000), (25_000,) * 20])
def test_piles(R, lengths, W, H):  # noqa: F811
    wl = piles(lengths, W, H)
    default, tile_first = check(R, wl, 1), check(R, wl, 0)
    imgs = [o["pb"].render_fwd() for o in (default, tile_first)]
    for k in imgs[0]:
        assert torch.equal(imgs[0][k], imgs[1][k]), k


@pytest.mark.parametrize("lengths", [(40_000, 9_000), (4_500, 300, 200)])
def test_piles_in_fewer_tiles_than_ctas_sort_them(R, lengths):  # noqa: F811
    check(R, piles(lengths, 32, 32, spread=100), 0)


def test_piles_twice_on_one_workspace(R):  # noqa: F811
    """The shared lists' tickets and counts start anew with every binning."""
    wl = piles((50_000, 20_000), 320, 240)
    got = check(R, wl, 0)
    for _ in range(3):
        got["pb"].project(got["g"])
        got["pb"].bin_sort()
        K = got["K"]
        assert got["pb"].check_status()[0] == 0
        np.testing.assert_array_equal(got["pb"].workspace()["sorted_vals"][:K].cpu().numpy().view(np.uint32), got["vals"])


def bin_us(wl):
    pb, g = gpu_problem(wl)
    times = []
    for _ in range(9):
        pb.project(g)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        ev[0].record()
        pb.bin_sort()
        ev[1].record()
        torch.cuda.synchronize()
        times.append(ev[0].elapsed_time(ev[1]) * 1e3)
    assert pb.check_status()[0] == 0
    return sorted(times)[4]


def test_a_pile_does_not_take_many_times_as_long(R):  # noqa: F811
    """400 k Gaussians in four tiles against the same number over the whole view, binned and sorted: one CTA per list
    made it 30 times as long, the shared sort 2 to 4 times."""
    assert bin_us(piles((100_000,) * 4, 640, 480)) < 8 * bin_us(piles((), 640, 480, spread=400_000))


def test_a_pile_does_not_wait_for_its_counters(R):  # noqa: F811
    """A million Gaussians in one tile: with an atomic per key on one counter the binning took 4.5 times as long as with
    the same number over the whole view, of which most was the wait for that counter; counted first, 1.5 times."""
    assert bin_us(piles((1_000_000,), 640, 480)) < 3 * bin_us(piles((), 640, 480, spread=1_000_000))

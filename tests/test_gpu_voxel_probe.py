"""Voxel sets keep blocks of voxels in lines of slots: every slot of every size of set can be reached, flat and
scattered sets alike, and membership agrees with what was inserted."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
V = 0.05


def _centres(kind, n, rng):
    """Centres of n distinct voxels, and the keys they must have."""
    if kind == "flat":        # a plane: one layer of each block
        side = int(np.ceil(np.sqrt(n)))
        i = np.stack(np.unravel_index(np.arange(n), (side, side)) + (np.full(n, 7),), 1) - 3
    elif kind == "far":       # beyond +-2^20 every index is the limit, so only y and z tell voxels apart
        i = np.stack((np.where(np.arange(n) % 2, 1 << 22, -(1 << 22)), np.arange(n) // 2, np.arange(n) % 5), 1)
    else:
        i = rng.permutation(200 ** 3)[:n]
        i = np.stack(np.unravel_index(i, (200, 200, 200)), 1) - 100
    x = ((i + 0.5) * V).astype(np.float32)
    idx = np.clip(np.floor(x / np.float32(V)).astype(np.int64), -(1 << 20), (1 << 20) - 1) + (1 << 20)
    keys = {(int(a) << 42) | (int(b) << 21) | int(c) for a, b, c in idx}
    assert len(keys) == n
    return torch.from_numpy(x).cuda(), keys


@pytest.mark.parametrize("kind", ["flat", "far", "scattered"])
@pytest.mark.parametrize("cap,n", [(2, 2), (4, 3), (8, 8), (16, 16), (32, 31), (64, 64), (1024, 1000), (1 << 14, 1 << 13)])
def test_every_slot_is_reached(kind, cap, n):
    from paper_2605_10760_gb300 import _lib as L, raster as R
    means, keys = _centres(kind, n + 1, np.random.default_rng(cap))
    small = torch.full((n + 1, 3), -12.0, device="cuda")     # boxes inside one voxel
    s = R.VoxSet(cap)
    s.add_boxes(means[:n], small[:n], 3.0, V)
    assert s.status() == (0, n)
    stored = s.keys()
    assert stored < keys
    keep = R.dedup_keep(means, s, None, V).cpu().numpy()
    assert not keep[:n].any() and keep[n] == 1
    s.add_boxes(means, small, 3.0, V)
    assert s.status() == ((0, n + 1) if n < cap else (L.GS_ERR_CAPACITY, n))


@pytest.mark.parametrize("n", [1, 31, 33, 300])
def test_boxes_of_uneven_sizes(n):
    from paper_2605_10760_gb300 import raster as R
    rng = np.random.default_rng(n)
    # half extents of a whole number of voxels minus a quarter around voxel centres: FP32 rounding cannot move a face
    half = rng.integers(1, 6, (n, 3))
    half[rng.random(n) < 0.1, 0] = 31                        # 63 voxels along one axis
    centre = rng.integers(-50, 50, (n, 3))
    means = torch.from_numpy(((centre + 0.5) * V).astype(np.float32)).cuda()
    logs = torch.from_numpy(np.log((half - 0.25) * V).astype(np.float32)).cuda()
    want = set()
    for c, h in zip(centre, half):
        r = [np.arange(c[a] - h[a], c[a] + h[a] + 1) + (1 << 20) for a in range(3)]
        # a half extent of h - 1/4 from the middle of voxel c reaches voxels c - h .. c + h when h - 1/4 > h - 1/2
        g = np.stack(np.meshgrid(*r, indexing="ij"), -1).reshape(-1, 3)
        want |= {(int(x) << 42) | (int(y) << 21) | int(z) for x, y, z in g}
    s = R.VoxSet(1 << 20)
    s.add_boxes(means, logs, 1.0, V)
    assert s.status() == (0, len(want)) and s.keys() == want


def test_an_overfull_set_reports_and_keeps_its_capacity():
    from paper_2605_10760_gb300 import _lib as L, raster as R
    cap = 1 << 12
    means, keys = _centres("scattered", 4 * cap, np.random.default_rng(1))
    small = torch.full((4 * cap, 3), -12.0, device="cuda")
    s = R.VoxSet(cap)
    for _ in range(2):
        s.add_boxes(means, small, 3.0, V)
        assert s.status() == (L.GS_ERR_CAPACITY, cap)
    assert s.keys() < keys
    keep = R.dedup_keep(means, s, None, V)
    assert int((keep == 0).sum()) == cap
    s.clear()
    s.add_boxes(means[:cap], small[:cap], 3.0, V)
    assert s.status() == (0, cap)

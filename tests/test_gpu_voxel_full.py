"""A voxel set that has no slot left says so and lets go of further keys soon, whatever was recorded before, and still
knows the keys it holds.  The times are bounds on the work: a surplus key tries a few dozen slots; if it walked the
set, or a sixteenth of it, the smaller set here would take a tenth of a second and the larger one several seconds."""
import time

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
V = 0.05


def centres(n, seed):
    """Centres of n distinct voxels of a cube, in random order."""
    side = int(np.ceil(n ** (1 / 3))) + 1
    i = np.random.default_rng(seed).permutation(side ** 3)[:n]
    i = np.stack(np.unravel_index(i, (side,) * 3), 1)
    return torch.from_numpy(((i + 0.5) * V).astype(np.float32)).cuda()


def timed(fn):
    torch.cuda.synchronize()
    t = time.perf_counter()
    fn()
    torch.cuda.synchronize()
    return time.perf_counter() - t


@pytest.mark.parametrize("wide_box_first", [False, True])
@pytest.mark.parametrize("cap,surplus,seconds", [(1 << 17, 10, 0.03), (1 << 22, 4, 0.3)])
def test_surplus_keys_do_not_walk_the_set(cap, surplus, seconds, wide_box_first):
    from paper_2605_10760_gb300 import _lib as L, raster as R
    means = centres(surplus * cap, cap)
    small = torch.full((len(means), 3), -12.0, device="cuda")
    s = R.VoxSet(cap)
    want = L.GS_ERR_CAPACITY
    if wide_box_first:     # an earlier error stays the recorded one
        s.add_boxes(means[:1], torch.full((1, 3), 2.0, device="cuda"), 3.0, V)
        want = L.GS_ERR_INVALID_ARG
        assert s.status() == (want, 0)
    assert timed(lambda: s.add_boxes(means, small, 3.0, V)) < seconds
    assert s.status() == (want, cap)
    assert timed(lambda: s.add_boxes(means, small, 3.0, V)) < seconds
    assert s.status() == (want, cap)


def test_surplus_rays_do_not_walk_the_set():
    from paper_2605_10760_gb300 import _lib as L, raster as R, scenes as S
    cap, h, w = 1 << 17, 340, 600
    cams = R.cameras_tensor([S.identity_camera(w, h, 300.0, 300.0)] * 4)
    depth = torch.full((4, h, w), 6.0, device="cuda")
    s = R.VoxSet(cap)
    assert timed(lambda: s.add_rays(cams, depth, 1, V)) < 0.1
    assert s.status() == (L.GS_ERR_CAPACITY, cap)


@pytest.mark.parametrize("cap", [2, 16, 1 << 10, 1 << 17])
def test_a_set_filled_to_the_last_slot_is_no_error(cap):
    from paper_2605_10760_gb300 import _lib as L, raster as R
    means = centres(cap + 64, 3)
    small = torch.full((len(means), 3), -12.0, device="cuda")
    s = R.VoxSet(cap)
    for part in (slice(0, cap // 2), slice(0, cap), slice(0, cap)):
        s.add_boxes(means[part], small[part], 3.0, V)
        assert s.status() == (0, len(means[part]))
    keep = R.dedup_keep(means, s, None, V).cpu().numpy()
    assert not keep[:cap].any() and keep[cap:].all()
    s.add_boxes(means[cap:], small[cap:], 3.0, V)
    assert s.status() == (L.GS_ERR_CAPACITY, cap)
    s.clear()
    s.add_boxes(means[:cap], small[:cap], 3.0, V)
    assert s.status() == (0, cap)


def test_asking_an_overfull_set_does_not_walk_it():
    """(A million absent keys against all four million stored ones would take minutes.)"""
    from paper_2605_10760_gb300 import _lib as L, raster as R
    cap, offered = 1 << 22, 9 << 19
    means = centres(offered + (1 << 20), 5)
    s = R.VoxSet(cap)
    s.add_boxes(means[:offered], torch.full((offered, 3), -12.0, device="cuda"), 3.0, V)
    assert s.status() == (L.GS_ERR_CAPACITY, cap)
    keep = torch.empty(len(means), dtype=torch.uint8, device="cuda")
    assert timed(lambda: keep.copy_(R.dedup_keep(means, s, None, V))) < 0.3
    assert int((keep == 0).sum()) == cap and bool(keep[offered:].all())

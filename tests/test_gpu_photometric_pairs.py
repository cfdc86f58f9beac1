"""The photometric kernel runs the chain of two pixels of a row at a time, 256 columns apart: rows shorter than one half, ending
inside either half and of a whole number of steps, with pixels without a depth (zero, negative, infinite, NaN) on
either side of a pair, and more edges than blocks are resident, against the FP64 sums over the pixels that the FP32
decisions keep (the tolerances of the synthetic edges)."""
import numpy as np
import pytest

from test_gpu_photometric import R, _compare, _synthetic  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,stride", [(2, 40, 1), (255, 9, 1), (256, 9, 1), (257, 9, 1), (511, 7, 1), (512, 7, 1),
                                        (513, 7, 1), (800, 6, 1), (1030, 12, 2)])
def test_rows_around_a_step_with_holes(R, W, H, stride):  # noqa: F811
    imgs, deps, cams, corrs = _synthetic(W, H, 7 * W + H)
    rng = np.random.default_rng(W)
    for k in (0, 1):
        for bad in (0.0, -1.0, np.inf, np.nan):
            deps[k][rng.random(deps[k].shape) < 0.08] = bad
    _compare(R, [(0, 1, 0, 1, 1.0), (1, 0, 1, 0, 0.5)], imgs, deps, cams, corrs, stride=stride)


def test_more_edges_than_resident_blocks(R):  # noqa: F811
    imgs, deps, cams, corrs = _synthetic(40, 12, 3)
    _compare(R, [(k % 2, 1 - k % 2, k % 4, (k + 1) % 4, 1.0 + k) for k in range(700)], imgs, deps, cams, corrs)

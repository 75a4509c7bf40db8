"""Image metrics at the sizes where their two paths and block shapes change.

Regions from none to more pixels than a block's shared memory holds, on and
off the image's edges, wider than the member list takes, more pairs than the
launch parameters hold, and values whose sums or squares leave FP32's range.
Whole numbers and the peak are exact; the others are doubles of well
conditioned sums of at most 2^18 terms, so 2^18 * 2^-53 < 3e-11 bounds any
order of summation, and 1e-12 is what the oracle comparison allows elsewhere
(both sides sum in parts of a few hundred terms)."""

import numpy as np
import pytest

from oracle import metrics as om
from test_gpu_metrics import _assert_same, _gpu_metrics

pytestmark = pytest.mark.gpu

GRID = dict(nx=420, nz=510, x0_m=-21e-3, x1_m=21e-3, z0_m=0.5e-3, z1_m=51.5e-3)  # 0.1 mm


def _disc(xc, zc, a):
    return dict(shape="disc", xc_m=xc * 1e-3, zc_m=zc * 1e-3, a_m=a * 1e-3)


def _ring(xc, zc, a, b):
    return dict(shape="annulus", xc_m=xc * 1e-3, zc_m=zc * 1e-3, a_m=a * 1e-3, b_m=b * 1e-3)


def _rect(xc, zc, a, b):
    return dict(shape="rect", xc_m=xc * 1e-3, zc_m=zc * 1e-3, a_m=a * 1e-3, b_m=b * 1e-3)


PAIRS = {
    "one_pixel": [(_disc(0.02, 20.02, 0.06), _ring(0, 20, 0.1, 0.16))],
    "block_steps": [(_disc(1, 20, r), _ring(1, 20, 1.3 * r, 1.9 * r)) for r in (1.5, 2.6, 3.8, 5.1, 7.3)],
    "at_the_limit": [(_disc(0, 26, 9.0), _ring(0, 26, 9.0, 14.0))],
    "beyond_it": [(_disc(0, 26, 9.0), _ring(0, 26, 9.5, 16.5))],
    "edges": [(_disc(-21, 0.5, 3), _ring(-21, 0.5, 3, 6)), (_disc(20.9, 51.4, 2), _ring(21, 51.5, 2.5, 5)),
              (_rect(-20, 30, 4, 3), _rect(19, 2, 5, 40)), (_disc(0, 26, 0), _ring(0, 26, 5, 4))],
    "thin": [(_rect(0, 20.02, 20, 0.04), _rect(3.02, 25, 0.04, 24)), (_rect(0, 26, 0.3, 25), _rect(0, 9, 20.9, 0.3))],
    "off_the_image": [(_disc(60, 20, 3), _disc(0, 20, 2)), (_disc(0, 20, 2), _rect(0, 90, 3, 3)),
                      (_disc(60, 20, 3), _rect(0, 90, 3, 3))],
    "more_than_the_parameters": [(_disc(-18 + i, 5 + 2 * i, 0.8), _ring(-18 + i, 5 + 2 * i, 1, 1.7))
                                 for i in range(17)],
}


@pytest.mark.parametrize("name", PAIRS)
def test_regions(name):
    rng = np.random.default_rng(7)
    images = rng.gamma(2.0, 1.0, (3, GRID["nx"], GRID["nz"])).astype(np.float32)
    images[1, 180:240, 190:290] += 9.0
    rois = PAIRS[name]
    _assert_same(_gpu_metrics(images, GRID, rois), om.metrics_batch(GRID, images, rois), name)


def test_wider_than_the_member_list():
    grid = dict(nx=1100, nz=40, x0_m=-55e-3, x1_m=55e-3, z0_m=0.0, z1_m=4e-3)
    images = np.random.default_rng(3).random((2, 1100, 40)).astype(np.float32)
    for half in (51.1, 51.2, 55.0):  # 1024 columns with their margin, and more
        rois = [(_disc(0, 2, 1), _rect(0, 2, half, 1.5))]
        _assert_same(_gpu_metrics(images, grid, rois), om.metrics_batch(grid, images, rois), half)


@pytest.mark.parametrize("scale", [1e-38, 1e-22, 1e-9, 1e18, 3e37])
def test_range_of_the_values(scale):
    """Sums above FP32's range and squares below it; a constant background."""
    rng = np.random.default_rng(5)
    images = (scale * rng.uniform(0.5, 10.0, (2, GRID["nx"], GRID["nz"]))).astype(np.float32)
    images[1, 200:, :] = np.float32(scale)
    rois = [(_disc(-3, 20, 2), _ring(-3, 20, 2.5, 4)), (_disc(-3, 20, 2), _disc(8, 20, 4))]
    g, r = _gpu_metrics(images, GRID, rois), om.metrics_batch(GRID, images, rois)
    # (the oracle's mean of equal values may differ from them in the last bit)
    assert g["sigma_out"][1, 1] == 0.0 and g["mu_out"][1, 1] == float(np.float32(scale))
    for f in ("sigma_out", "snr_db"):
        r[f][1, 1] = g[f][1, 1]
    _assert_same(g, r, scale)


def test_nearly_constant_background():
    """Deviations of one unit in the last place around the mean."""
    images = np.full((1, GRID["nx"], GRID["nz"]), 3.0, np.float32)
    images[0, ::3, ::2] = np.nextafter(np.float32(3.0), np.float32(4.0))
    rois = [(_disc(0, 20, 2), _ring(0, 20, 2.5, 4))]
    g = _gpu_metrics(images, GRID, rois)
    m = om.region_mask(GRID, rois[0][1])
    up = np.count_nonzero(images[0][m] > 3.0) / np.count_nonzero(m)
    assert g["sigma_out"][0, 0] == pytest.approx(2.0**-22 * np.sqrt(up * (1 - up)), rel=1e-12)


def test_infinities_and_nan_in_the_background():
    """The sums take them as FP64 sums do."""
    images = np.random.default_rng(9).random((3, GRID["nx"], GRID["nz"])).astype(np.float32)
    rois = [(_disc(0, 20, 2), _ring(0, 20, 2.5, 4))]
    j, l = np.argwhere(om.region_mask(GRID, rois[0][1]))[100]
    images[0, j, l], images[1, j, l], images[2, j, l] = np.inf, -np.inf, np.nan
    g = _gpu_metrics(images, GRID, rois)
    assert g["mu_out"][0, 0] == np.inf and g["mu_out"][1, 0] == -np.inf and np.isnan(g["mu_out"][2, 0])
    assert np.isnan(g["sigma_out"]).all() and np.isfinite(g["mu_in"]).all()

"""Scalar extraction at the sizes where its kernels change over, against the
oracle: level counts around the eigen-solver's shared-memory rows (64 / 65) and
the triangle's odd and even row pairing up to 255 levels, histograms of one bin
and of the whole 16-bit range, one voxel, and sparse masks.  The bar is the
scalar maps': 1e-8 max(1, |oracle|), MCC max(1e-6, 1e-4 |oracle|)."""
import numpy as np
import pytest

from test_gpu_scalar import ALL, _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("merged", [False, True])
@pytest.mark.parametrize("nlev", [1, 2, 3, 24, 31, 32, 63, 64, 65, 66, 200, 255])
def test_level_counts(nlev, merged):
    rng = np.random.default_rng(nlev)
    img = rng.integers(0, nlev, size=(9, 10, 13)).astype(np.int16)
    img.flat[0], img.flat[1] = 0, nlev - 1
    kw = dict(aggregation=int(merged))
    _check(img, np.ones(img.shape, np.uint8), disc_mode=0, bin_count=nlev, features=ALL, **kw)


@pytest.mark.parametrize("fill", [0.0, 0.02, 0.5, 1.0])
@pytest.mark.parametrize("lo, hi", [(7, 7), (-32768, 32767), (-1000, 1100)])
def test_histogram_ranges(lo, hi, fill):
    rng = np.random.default_rng(hi - lo)
    img = rng.integers(lo, hi + 1, size=(11, 9, 14)).astype(np.int16)
    mask = (rng.random(img.shape) < fill).astype(np.uint8)
    mask[5, 4, 6] = 1
    _check(img, mask, disc_mode=0, bin_count=17, features=ALL)

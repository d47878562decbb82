"""The window and first-order paths of the mapping kernel where one hands over
to the next, against the oracle: intensity spans around 4,096 (power sums in
64 bits / general sums) with the two-sided windows whose fourth power sums are
largest, 343 / 729 keys, the counting sort of 9^3 and larger windows up to the
bin limit, and masks that leave few of a padded window's voxels.  Tolerance:
the maps' bar, |gpu - oracle| <= max(1e-6, 1e-4 |oracle|)."""
import numpy as np
import pytest

import gpu_helpers as H
import parity
from oracle import oracle as O

pytestmark = pytest.mark.gpu

FEATS = list(range(93))


def _check(img, mask, r, **kw):
    kw = dict(disc_mode=0, bin_count=12, kernel_radius=r, **kw)
    got, plan, feats = H.gpu_map(img, mask, features=FEATS, **kw)
    ref, _, _, _ = H.oracle_map(img, mask, **kw)
    parity.assert_close(got, ref[feats], [O.feature_names()[f] for f in feats])


@pytest.mark.parametrize("r", [1, 3, 4])
@pytest.mark.parametrize("span", [1, 4094, 4095, 4096, 65535])
@pytest.mark.parametrize("share", [0.02, 0.5, 0.98])
def test_intensity_span(r, span, share):
    # two intensities `span` apart (and a few between) in shares share : 1 - share
    rng = np.random.default_rng(span + r)
    img = np.where(rng.random((6, 7, 8)) < share, span, 0)
    few = rng.random(img.shape) < 0.05
    img = np.where(few, rng.integers(0, span + 1, img.shape), img)
    img.flat[0], img.flat[1] = 0, span
    _check((img - 32768 + (0 if span == 65535 else 31768)).astype(np.int16),
           np.ones(img.shape, np.uint8), r)


@pytest.mark.parametrize("r", [2, 4, 5, 6, 7])
@pytest.mark.parametrize("span", [40, 1200, 30000])
@pytest.mark.parametrize("fill", [0.08, 0.6, 1.0])
def test_large_windows(r, span, fill):
    rng = np.random.default_rng(100 * r + span)
    img = rng.integers(-1000, span - 1000, size=(7, 6, 9)).astype(np.int16)
    mask = (rng.random(img.shape) < fill).astype(np.uint8)
    mask[3, 3, 4] = 1
    _check(img, mask, r)


@pytest.mark.parametrize("r", [2, 4])
def test_distance_two_large(r):
    rng = np.random.default_rng(r)
    img = rng.integers(0, 300, size=(7, 8, 9)).astype(np.int16)
    _check(img, (rng.random(img.shape) < 0.7).astype(np.uint8), r, glcm_distance=2)

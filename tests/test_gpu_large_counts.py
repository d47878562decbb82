"""Windows of many pairs, against the oracle: merged GLCM and GLRLM matrices of
sides 9 to 15, where a filled window's pair total passes 2^12 (its square the
integers of fp32) and, from side 13 on, 46,341 (its square 2^31); and side 15 per
direction.  Levels of near-symmetric distribution: ClusterShade is the small
mean of values of either sign.  Tolerance: the maps' bar, |gpu - oracle| <=
max(1e-6, 1e-4 |oracle|)."""
import numpy as np
import pytest

import gpu_helpers as H
import parity
from oracle import oracle as O

pytestmark = pytest.mark.gpu

ALL = list(range(101))


def _check(r, nlev, seed, fill, **kw):
    rng = np.random.default_rng(seed)
    shape = (2 * r + 1, 2 * r + 2, 2 * r + 3)
    img = rng.integers(0, nlev, size=shape).astype(np.int16)
    img.flat[0], img.flat[1] = 0, nlev - 1
    mask = (rng.random(shape) < fill).astype(np.uint8)
    mask[r, r, r] = 1
    kw = dict(disc_mode=0, bin_count=nlev, kernel_radius=r, **kw)
    allvox = np.flatnonzero(mask.reshape(-1))
    centre = (r * shape[1] + r) * shape[2] + r  # its window is the whole image but a rim
    voxels = np.unique(np.append(rng.choice(allvox, 40, replace=False), centre)).astype(np.int64)
    got, _, feats = H.gpu_map(img, mask, features=ALL, **kw)
    ref, _, _, _ = H.oracle_map(img, mask, voxels=voxels, **kw)
    parity.assert_close(got[:, np.searchsorted(allvox, voxels)], ref[feats],
                        [O.feature_names()[f] for f in feats])


@pytest.mark.parametrize("nlev", [2, 16, 64])
@pytest.mark.parametrize("r", [3, 4, 5, 6, 7])
def test_merged(r, nlev):
    _check(r, nlev, 10 * r + nlev, 1.0, aggregation=1)


@pytest.mark.parametrize("fill", [0.6, 1.0])
@pytest.mark.parametrize("nlev", [2, 16, 64])
def test_side_fifteen(nlev, fill):
    _check(7, nlev, nlev, fill)


@pytest.mark.parametrize("kw", [dict(), dict(glcm_distance=2), dict(aggregation=1)])
@pytest.mark.parametrize("share", [0.21, 0.5, 0.98])
@pytest.mark.parametrize("r", [3, 7])
def test_widest_span(r, share, kw):
    # two levels 254 apart (and a few between): the largest power sums and
    # third moments of the class sums (a share of 0.21 has the largest)
    rng = np.random.default_rng(r)
    shape = (2 * r + 1, 2 * r + 2, 2 * r + 3)
    img = np.where(rng.random(shape) < share, 254, 0)
    img = np.where(rng.random(shape) < 0.02, rng.integers(0, 255, shape), img).astype(np.int16)
    img.flat[0], img.flat[1] = 0, 254
    kw = dict(disc_mode=0, bin_count=255, kernel_radius=r, **kw)
    voxels = np.unique(np.append(rng.choice(img.size, 24, replace=False),
                                 (r * shape[1] + r) * shape[2] + r)).astype(np.int64)
    mask = np.ones(shape, np.uint8)
    got, _, feats = H.gpu_map(img, mask, features=ALL, **kw)
    ref, _, _, _ = H.oracle_map(img, mask, voxels=voxels, **kw)
    parity.assert_close(got[:, voxels], ref[feats], [O.feature_names()[f] for f in feats])

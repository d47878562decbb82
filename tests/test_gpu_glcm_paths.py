"""The GLCM paths of the mapping kernel at the sizes where one hands over to
the next, against the oracle: level counts around the lanes-by-direction
limit (15 / 16), the shared-memory limit (24 / 25 levels, level range 63 / 64),
the triangle and hash tables (31 / 32) and the register solve (48), a level
with more voxels than a byte counts (7^3 windows), and level graphs that are
bipartite or disconnected (MCC exactly 1).  Tolerance: the maps' bar,
|gpu - oracle| <= max(1e-6, 1e-4 |oracle|); counts bit-exact."""
import numpy as np
import pytest

import gpu_helpers as H
import parity
from oracle import oracle as O

pytestmark = pytest.mark.gpu

FEATS = list(range(93))


def _check(img, nlev, r, **kw):
    mask = np.ones(img.shape, np.uint8)
    kw = dict(disc_mode=0, bin_count=nlev, kernel_radius=r, **kw)
    got, plan, feats = H.gpu_map(img, mask, features=FEATS, **kw)
    ref, _, _, _ = H.oracle_map(img, mask, **kw)
    parity.assert_close(got, ref[feats], [O.feature_names()[f] for f in feats])


def _noise(shape, nlev, seed):
    """Uniform levels 0..nlev-1, both ends present (FBN nlev keeps them apart)."""
    rng = np.random.default_rng(seed)
    img = rng.integers(0, nlev, size=shape).astype(np.int16)
    img.flat[0], img.flat[1] = 0, nlev - 1
    return img


@pytest.mark.parametrize("r", [1, 2, 3])
@pytest.mark.parametrize("nlev", [1, 2, 4, 8, 12, 13, 15, 16, 17, 24, 25, 31, 32, 48, 64, 65, 100])
def test_level_counts(r, nlev):
    _check(_noise((6, 7, 9), nlev, 100 * r + nlev), nlev, r)


@pytest.mark.parametrize("others", [3, 9, 10, 14])
def test_dominant_level(others):
    # 7^3 windows with one level over 255 voxels: 16-bit cells up to 10
    # levels, the general path beyond
    img = np.zeros((7, 8, 9), np.int16)
    rng = np.random.default_rng(others)
    at = rng.choice(img.size, 60, replace=False)
    img.flat[at] = 1 + np.arange(60) % others
    _check(img, others + 1, 3)


@pytest.mark.parametrize("r", [1, 2, 3])
@pytest.mark.parametrize("span", [63, 64, 200])
def test_level_range(r, span):
    # few levels, far apart: class sums by number, and the range limit of the
    # shared-memory region
    img = _noise((6, 7, 8), 6, span)
    _check((img.astype(np.int32) * span // 5).astype(np.int16), span + 1, r)


@pytest.mark.parametrize("nlev", [6, 30, 64])
def test_distance_two(nlev):
    _check(_noise((6, 7, 8), nlev, nlev), nlev, 2, glcm_distance=2)


@pytest.mark.parametrize("r", [1, 2])
def test_bipartite_and_disconnected(r):
    # levels of one parity on each colour of a checkerboard (bipartite along
    # the axes, disconnected along the face diagonals), more than 24 of them
    rng = np.random.default_rng(5)
    z, y, x = np.indices((6, 7, 8))
    img = (2 * rng.integers(0, 30, size=(6, 7, 8)) + (z + y + x) % 2).astype(np.int16)
    img.flat[0], img.flat[1] = 0, 59
    _check(img, 60, r)

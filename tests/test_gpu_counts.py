"""Integer texture matrices of the mapping kernel, bit-exact against the oracle,
on every counting path of the GLCM and the families after it: level counts
around the limits of the direction lanes (15 / 16), the shared region (24 / 25)
and the triangle and hash tables (31 / 32); levels of more than 255 voxels;
windows that are mostly empty (cell (0, 0) of a byte table passes 255); distance
2; merged matrices; windows of side 9."""
import numpy as np
import pytest
import torch

import gpu_helpers as H
import paper_2609_19190_gb300 as fm
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _check(img, mask, nlev, r, n=24, **kw):
    kw = dict(disc_mode=0, bin_count=nlev, kernel_radius=r, **kw)
    _, plan, _ = H.gpu_map(img, mask, **kw)
    op = H.oracle_params(img.shape, **kw)
    levels, ng, _, _ = O.discretise(op, img, mask)
    allvox = np.flatnonzero(mask.reshape(-1))
    cols = np.unique(np.linspace(0, allvox.size - 1, n).astype(np.int32))
    m = fm.fr_debug_matrices(plan, torch.from_numpy(img).cuda(), cols, ng)
    for t, c in enumerate(cols):
        ref = O.matrices(op, levels, ng, int(allvox[c]))
        if kw.get("aggregation"):  # one matrix for the 13 directions
            for key in ("glcm", "glrlm"):
                assert np.array_equal(m[key][t][0], ref.pop(key).sum(0)), (key, t, c)
        for key in ref:
            assert np.array_equal(m[key][t], ref[key]), (key, t, c)
        assert m["nv"][t] == ref["hist"].sum()


def _noise(nlev, seed, shape=(8, 9, 10)):
    rng = np.random.default_rng(seed)
    img = rng.integers(0, nlev, size=shape).astype(np.int16)
    img.flat[0], img.flat[1] = 0, nlev - 1
    return img, rng


@pytest.mark.parametrize("r", [1, 2, 3, 4])
@pytest.mark.parametrize("nlev", [1, 2, 12, 13, 15, 16, 24, 25, 31, 32, 64, 100])
def test_levels(r, nlev):
    img, _ = _noise(nlev, 10 * nlev + r)
    _check(img, np.ones(img.shape, np.uint8), nlev, r)


@pytest.mark.parametrize("others", [3, 9, 10, 14])
def test_dominant_level(others):
    img, rng = _noise(1, others)
    at = rng.choice(img.size, 70, replace=False)
    img.flat[at] = 1 + np.arange(70) % others
    _check(img, np.ones(img.shape, np.uint8), others + 1, 3)


@pytest.mark.parametrize("r", [1, 2, 3, 4])
@pytest.mark.parametrize("nlev", [3, 14, 40])
@pytest.mark.parametrize("fill", [0.02, 0.1, 0.5])
def test_sparse_masks(r, nlev, fill):
    img, rng = _noise(nlev, 1000 * r + nlev)
    mask = (rng.random(img.shape) < fill).astype(np.uint8)
    mask.flat[[0, 1]] = 1
    mask[4, 4, 5] = 1
    _check(img, mask, nlev, r)


@pytest.mark.parametrize("r", [1, 2, 3, 4])
@pytest.mark.parametrize("nlev", [6, 24, 40])
@pytest.mark.parametrize("kw", [dict(glcm_distance=2), dict(aggregation=1)])
def test_distance_and_merged(r, nlev, kw):
    img, rng = _noise(nlev, 77 * r + nlev)
    _check(img, (rng.random(img.shape) < 0.8).astype(np.uint8) | (img == nlev - 1) | (img == 0),
           nlev, r, **kw)

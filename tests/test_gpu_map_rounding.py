"""How far fp32 maps of exact integer numerators are from 64 bits.

A feature that is an exact integer over a power of a direction's total is
rounded a known number of times.  Independent roundings to nearest of a value
with mantissa 1 have a relative rms of 2^-24 / sqrt(3) each, so k of them at most
sqrt(k) times that over a map (2-norm of the difference over 2-norm of the map).
k counts at most the numerator, the reciprocal of the total's power, the product, the
sum over directions, and two for the division by their number; a numerator of
128 bits is rounded twice, and T^4 itself once."""
import math

import numpy as np
import pytest

import gpu_helpers as H
from oracle import oracle as O
from paper_2609_19190_gb300 import synth

pytestmark = pytest.mark.gpu

NAMES = {n: i for i, n in enumerate(O.feature_names())}
GLCM = {"glcm_ClusterTendency": 6, "glcm_DifferenceVariance": 6, "glcm_JointEnergy": 6,
        "glcm_SumSquares": 6, "glcm_SumVariance": 6, "glcm_ClusterProminence": 8}
GLRLM = {"glrlm_GrayLevelNonUniformityNormalized": 6, "glrlm_RunLengthNonUniformityNormalized": 6,
         "glrlm_GrayLevelVariance": 6, "glrlm_RunVariance": 6}


def _distances(names, shape, r, **kw):
    img = synth.ct_like(shape, 5)
    mask = synth.ellipsoid(shape, tuple((n - 1) / 2 for n in shape[::-1]),
                           tuple(0.47 * n for n in shape[::-1]))
    kw = dict(kernel_radius=r, **kw)
    ids = sorted(NAMES[n] for n in names)
    got, _, _ = H.gpu_map(img, mask, features=ids, **kw)
    ref = H.oracle_map(img, mask, **kw)[0][ids]
    inv = {i: n for n, i in NAMES.items()}
    out = {}
    for k, i in enumerate(ids):
        ok = np.isfinite(ref[k])
        out[inv[i]] = np.linalg.norm(got[k][ok] - ref[k][ok]) / np.linalg.norm(ref[k][ok])
    return out


def _check(names, shape, r, **kw):
    far = _distances(names, shape, r, **kw)
    bad = {n: (far[n], math.sqrt(k / 3.0) * 2.0 ** -24) for n, k in names.items()
           if not far[n] <= math.sqrt(k / 3.0) * 2.0 ** -24}
    assert not bad, bad


WINDOWS = pytest.mark.parametrize("r, disc", [(1, dict(disc_mode=1, bin_width=25.0)),
                                              (2, dict(disc_mode=1, bin_width=25.0)),
                                              (3, dict(disc_mode=0, bin_count=64))])


@WINDOWS
def test_glcm(r, disc):
    _check(GLCM, (20, 24, 28), r, **disc)


@WINDOWS
def test_glrlm(r, disc):
    _check(GLRLM, (20, 24, 28), r, **disc)

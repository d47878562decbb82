"""MCC of scalar extraction where it is small, against the oracle.  The matrix
A = S - u u^T is rounded to fp32 and reduced by n - 2 reflections in fp32, so the
largest |eigenvalue| is known to n 2^-24 |A|_F (each reflection and the rounding
of the elements move it by about 2^-24 |A|_F).  Independent levels keep |A|_F
far below 1: the solver has to refine to the scale of A, not to an absolute
width."""
import numpy as np
import pytest

from oracle import oracle as O
from test_gpu_scalar import MCC, _gpu_scalar, _oracle_scalar

pytestmark = pytest.mark.gpu


def _shift(a, d):
    """The part of `a` that has a neighbour at -d (aligned with _shift(a, -d))."""
    return a[tuple(slice(max(k, 0), n + min(k, 0)) for k, n in zip(d, a.shape))]


def _norm(img, nlev):
    """|S - u u^T|_F of the merged matrix of the whole volume."""
    c = np.zeros((nlev, nlev))
    for d in O.directions():
        d = tuple(int(k) for k in d)
        np.add.at(c, (_shift(img, tuple(-k for k in d)), _shift(img, d)), 1.0)
    c += c.T
    p = c / c.sum()
    px = p.sum(1)
    u = np.sqrt(px)
    return np.linalg.norm(p / np.outer(u, u) - np.outer(u, u))


@pytest.mark.parametrize("nlev", [8, 16, 24, 40, 64])
@pytest.mark.parametrize("side", [11, 13, 16, 20, 25, 31, 39])
def test_independent_levels(nlev, side):
    rng = np.random.default_rng(100 * nlev + side)
    img = rng.integers(0, nlev, size=(side, side + 1, side + 2)).astype(np.int16)
    img.flat[0], img.flat[1] = 0, nlev - 1
    kw = dict(disc_mode=0, bin_count=nlev, aggregation=1)
    mask = np.ones(img.shape, np.uint8)
    got, _ = _gpu_scalar(img, mask, features=[MCC], **kw)
    ref = _oracle_scalar(img, mask, **kw)[MCC]
    assert abs(got[0] - ref) <= nlev * 2.0 ** -24 * _norm(img, nlev)

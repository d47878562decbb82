"""MCC of windows whose level matrix has nearly all eigenvalues in one place,
against the oracle: every pair of n levels meets equally often (and every level
itself equally often), so S - u u^T has one eigenvalue n - 1 times, and the
characteristic polynomial next to it is a product of as many small factors.

The VOI is a set of rows along x, two apart in y and z, so that only x has
pairs, and the rows are the pieces of Euler trails of the complete graph of the
levels.  Row counts of the solvers: 4, 8, 12 (a matrix per lane), 16 (four lanes
each), 24 (a warp each).  Tolerance: the maps' bar, |gpu - oracle| <=
max(1e-6, 1e-4 |oracle|)."""
import random

import numpy as np
import pytest

import gpu_helpers as H
import parity
from oracle import oracle as O

pytestmark = pytest.mark.gpu

MCC = 41


def _trails(n, loops, rng):
    """The complete graph on n levels (with `loops` loops a level) as trails:
    an Euler circuit, for even n cut at an added perfect matching."""
    adj = {a: [(b, False) for b in range(n) if b != a] + [(a, False)] * loops for a in range(n)}
    if n % 2 == 0:
        for a in range(n):
            adj[a].append((a ^ 1, True))
    for a in adj:
        rng.shuffle(adj[a])

    def take(a):
        b, extra = adj[a].pop()
        if b != a:
            adj[b].remove((a, extra))
        return b, extra

    stack, circuit = [(0, False)], []
    while stack:
        a, _ = stack[-1]
        if adj[a]:
            stack.append(take(a))
        else:
            circuit.append(stack.pop())
    trails = [[circuit[0][0]]]
    for (_, extra), (b, _) in zip(circuit, circuit[1:]):
        if extra:
            trails.append([b])
        else:
            trails[-1].append(b)
    if n % 2 == 0:  # the circuit closes inside a trail
        trails[0] = trails.pop() + trails[0][1:]
    return trails


def _rows(n, loops, side, places):
    """Rows of at most `side` levels, no more than there are places."""
    for seed in range(100000):
        rows = [t[k:k + side] for t in _trails(n, loops, random.Random(seed))
                for k in range(0, len(t) - 1, side - 1)]
        if len(rows) <= places:
            return rows
    raise AssertionError("the rows do not fit")


def _places(r):
    """(z, y) of rows two apart in a window of radius r, its centre among them."""
    if r == 3:  # 11 rows hold the 66 pairs of 12 levels
        return [(z, y) for z in (1, 3, 5) for y in range(1 if z == 3 else 0, 7, 2)]
    return [(z, y) for z in range(r % 2, 2 * r + 1, 2) for y in range(r % 2, 2 * r + 1, 2)]


def _volume(n, loops, r):
    side = 2 * r + 1
    places = _places(r)
    rows = sorted(_rows(n, loops, side, len(places)), key=len, reverse=True)
    places.sort(key=lambda p: p != (r, r))  # the centre gets a whole row
    img = np.zeros((side, side, side), np.int16)
    mask = np.zeros(img.shape, np.uint8)
    for (z, y), row in zip(places, rows):
        img[z, y, :len(row)] = row
        mask[z, y, :len(row)] = 1
    assert mask[r, r, r]
    return img, mask


def _check(n, loops, r, **kw):
    img, mask = _volume(n, loops, r)
    kw = dict(disc_mode=0, bin_count=n, kernel_radius=r, **kw)
    ref, vox, _, _ = H.oracle_map(img, mask, **kw)
    centre = int(np.flatnonzero(vox == img.size // 2)[0])
    # S = (1 / c) (J - I + 2 loops I), c = n - 1 + 2 loops: the window is the
    # whole matrix
    assert abs(ref[MCC, centre] - abs(2 * loops - 1) / (n - 1 + 2 * loops)) < 1e-12
    got, _, feats = H.gpu_map(img, mask, features=list(range(18, 42)), **kw)
    parity.assert_close(got, ref[feats], [O.feature_names()[f] for f in feats])


@pytest.mark.parametrize("n", [9, 11, 12])
def test_side_seven(n):
    _check(n, 0, 3)


@pytest.mark.parametrize("merged", [0, 1])
@pytest.mark.parametrize("loops", [0, 1, 3])
@pytest.mark.parametrize("n", [4, 5, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16])
def test_up_to_sixteen_rows(n, loops, merged):
    _check(n, loops, 4, aggregation=merged)


@pytest.mark.parametrize("loops", [0, 1])
@pytest.mark.parametrize("n", [17, 18, 19, 20, 21, 22, 23, 24])
def test_seventeen_rows_and_more(n, loops):
    _check(n, loops, 6)

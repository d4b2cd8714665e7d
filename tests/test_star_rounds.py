"""The star path's rule in whole numbers on the CPU: candidates in angular
order about a point c, rounds that drop a point inside the triangle of c and
its two neighbours, and the verification of what is left.  Whenever the
verification accepts, the polygon must be the oracle's hull, whatever c is
and however the points were ordered inside float rounding; on ordinary sets
it must accept."""
import functools

import numpy as np
import pytest

import oracle


def cross(a, b):
    return a[0] * b[1] - a[1] * b[0]


def half(p):
    return 0 if (p[1] > 0 or (p[1] == 0 and p[0] > 0)) else 1


def star_hull(pts, c, swap=None, strict_verify=True):
    """Indices of the hull, or None when it does not verify."""
    rel = [(int(x) - c[0], int(y) - c[1]) for x, y in pts]

    def less(i, j):
        a, b = rel[i], rel[j]
        if half(a) != half(b):
            return half(a) - half(b)
        k = cross(a, b)
        if k:
            return -1 if k > 0 else 1
        da, db = abs(a[0]) + abs(a[1]), abs(b[0]) + abs(b[1])
        return db - da if da != db else i - j

    live = sorted((i for i in range(len(pts)) if rel[i] != (0, 0)), key=functools.cmp_to_key(less))
    order = []
    for i in live:                       # the first of every ray
        if not order or half(rel[order[-1]]) != half(rel[i]) or cross(rel[order[-1]], rel[i]) != 0:
            order.append(i)
    if swap is not None and len(order) > 3:
        k = swap % (len(order) - 1)
        order[k], order[k + 1] = order[k + 1], order[k]
    while len(order) >= 3:
        m, kept, good = len(order), [], True
        for k in range(m):
            a, q, b = rel[order[k - 1]], rel[order[k]], rel[order[(k + 1) % m]]
            ab, aq, qb = cross(a, b), cross(a, q), cross(q, b)
            o = ab - aq - qb
            if not (ab > 0 and aq >= 0 and qb >= 0 and (o > 0 or (o == 0 and aq > 0 and qb > 0))):
                kept.append(order[k])
            good = good and aq > 0 and qb > 0 and o < 0
        if len(kept) == m:
            if strict_verify and not good:
                return None
            s = min(range(m), key=lambda k: (int(pts[order[k]][0]), int(pts[order[k]][1])))
            return order[s:] + order[:s]
        order = kept
    return None


def some_sets(count, seed):
    rng = np.random.default_rng(seed)
    for _ in range(count):
        n = int(rng.integers(3, 60))
        r = int(rng.choice([2, 5, 30, 1 << 29]))
        pts = rng.integers(-r, r + 1, size=(n, 2)).astype(np.int32)
        kind = rng.integers(0, 4)
        if kind == 1:
            pts[:, 1] = pts[:, 0] // 2          # nearly on a line
        elif kind == 2:
            pts[n // 2:] = pts[: n - n // 2]    # duplicates
        yield rng, pts


@pytest.mark.parametrize("seed", range(4))
def test_verified_means_hull(seed):
    accepted = total = 0
    for rng, pts in some_sets(400, seed):
        ref = oracle.hull(pts).tolist()
        mean = tuple(int(v) for v in np.rint(pts.astype(np.float64).mean(axis=0)))
        got = star_hull(pts, mean)
        total += 1
        accepted += got is not None
        assert got is None or got == ref
        # A c anywhere (a corner, outside) and a misplaced pair: refused or right.
        far = tuple(int(v) for v in rng.integers(-40, 41, size=2))
        for c in (tuple(int(v) for v in pts[0]), far):
            got = star_hull(pts, c)
            assert got is None or got == ref
        got = star_hull(pts, mean, swap=int(rng.integers(0, 60)))
        assert got is None or got == ref
    assert accepted > total // 2


def test_without_the_verification_it_would_be_wrong():
    wrong = 0
    for rng, pts in some_sets(400, 9):
        got = star_hull(pts, tuple(int(v) for v in pts[0]), strict_verify=False)
        wrong += got is not None and got != oracle.hull(pts).tolist()
    assert wrong > 0

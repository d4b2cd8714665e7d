"""The star path's frame and angular bins (csrc/star.cuh: frame_of, to_uv,
bin_of) in 32-bit floats on the CPU.  The verification of the star path's
polygon is local (a pentagram passes it), so the list that it looks at has to
go round once: the map must stay bounded whatever its sums lost to rounding,
and the bins must be one sweep of the exact angle."""
import math

import numpy as np
import pytest

f32 = np.float32
ONE = 1 << 29


def frame(sample, o):
    """(cx, cy, m00, m10, m11), the sums in pairs as a block reduces them."""
    fx, fy = sample[:, 0].astype(f32) - f32(o[0]), sample[:, 1].astype(f32) - f32(o[1])

    def mean(v):
        v = v.astype(f32)
        while len(v) > 1:
            v = v[0::2] + v[1::2]
        return v[0] * f32(1.0 / len(sample))

    mx, my = mean(fx), mean(fy)
    a, d = max(mean(fx * fx) - mx * mx, f32(1)), max(mean(fy * fy) - my * my, f32(1))
    b = mean(fx * fy) - mx * my
    l11, sd = np.sqrt(a), np.sqrt(d)
    l21 = min(max(b / l11, -sd), sd)
    l22 = np.sqrt(max(d - l21 * l21, f32(1.0e-8) * d))
    c = [int(np.rint(min(max(f32(o[k]) + m, f32(-ONE)), f32(ONE)))) for k, m in ((0, mx), (1, my))]
    return c[0], c[1], f32(1) / l11, -(l21 / l11) / l22, f32(1) / l22


def bins(F, pts, nb):
    fx, fy = (pts[:, 0] - F[0]).astype(f32), (pts[:, 1] - F[1]).astype(f32)
    u = fx * F[2]
    v = (fy.astype(np.float64) * np.float64(F[4]) + (fx * F[3]).astype(np.float64)).astype(f32)   # one rounding: fma
    with np.errstate(invalid="ignore"):
        t = v / (np.abs(u) + np.abs(v))
    a = np.where(u >= 0, np.where(v >= 0, t, f32(4) + t), f32(2) - t)
    return np.clip(np.nan_to_num(a * f32(nb // 4)).astype(np.int64), 0, nb - 1)


def sets():
    rng = np.random.default_rng(3)
    n = 4096
    for k in range(40):
        r = int(rng.integers(1, 1 << int(rng.integers(1, 29))))
        p = rng.integers(-r, r + 1, size=(n, 2)).astype(np.int64)
        kind = k % 4
        if kind == 1:                      # a tight set far from the sample's first point
            at = rng.integers(-ONE + r, ONE - r, size=2)
            p = p + at
            p[0] = -np.sign(at) * ONE
        elif kind == 2:                    # a needle along a diagonal
            t = rng.integers(-ONE + 8, ONE - 8, size=n)
            p = np.stack([t, np.clip(t // int(rng.integers(1, 9)) + rng.integers(-3, 4, size=n), -ONE, ONE)], axis=1)
        elif kind == 3:                    # one or two columns
            p = np.stack([rng.integers(0, 2, size=n), rng.integers(-ONE, ONE, size=n)], axis=1)
        yield p


@pytest.mark.parametrize("nb", [512, 2048, 1 << 16])
def test_bins_are_one_sweep(nb):
    for p in sets():
        F = frame(p, p[0])
        assert abs(F[3]) <= 1.0001e4 * F[2]
        q = p[(p[:, 0] != F[0]) | (p[:, 1] != F[1])]
        b = bins(F, q, nb)
        # The whitened angle without rounding, against the bin's own interval.
        dx, dy = (q[:, 0] - F[0]).astype(np.longdouble), (q[:, 1] - F[1]).astype(np.longdouble)
        ang = np.arctan2((dy * F[4] + dx * F[3]).astype(float), (dx * F[2]).astype(float)) % (2 * math.pi)

        def edge(k):                       # the angle of diamond parameter 4 k / nb
            a = 4.0 * k / nb
            s, r = int(a) % 4, a - int(a)
            x, y = ((1 - r, r), (-r, 1 - r), (r - 1, -r), (r, r - 1))[s]
            return math.atan2(y, x) % (2 * math.pi)

        lo = np.array([edge(k) for k in range(nb)])
        off = (ang - lo[b] + math.pi) % (2 * math.pi) - math.pi
        assert off.min() > -2.0 ** -8 and off.max() < 2.0 ** -8 + 2 * math.pi * 2 / nb


def test_a_pentagram_passes_the_local_tests():
    """Why the sweep is needed: two turns, every local test passed."""
    p = [(round(1000 * math.cos(4 * math.pi * k / 5)), round(1000 * math.sin(4 * math.pi * k / 5))) for k in range(5)]
    for k in range(5):
        a, q, b = p[k - 1], p[k], p[(k + 1) % 5]
        aq, qb, ab = (s[0] * t[1] - s[1] * t[0] for s, t in ((a, q), (q, b), (a, b)))
        assert aq > 0 and qb > 0 and ab - aq - qb < 0

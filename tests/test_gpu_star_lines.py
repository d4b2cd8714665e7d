"""Large inputs without a sample polygon because the sample lies on one line or
on one point: the pass keeps each warp's extremes of that line and every point
off it.  Whole lines, lines with a few points off them (between the sampled
ones), duplicates, range limits, odd rows, single and batched."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ONE = 1 << 29
STEPS = {"flat": (1, 0), "up": (0, 1), "diagonal": (3, 5), "falling": (7, -2), "point": (0, 0)}


def line(kind, n, seed):
    """n points on a line in random order, a third of them equal to others."""
    rng = np.random.default_rng(seed)
    dx, dy = STEPS[kind]
    reach = min(n, (ONE - 100) // max(abs(dx), abs(dy), 1))
    t = rng.integers(-reach, reach + 1, size=n)
    t[n // 3: 2 * (n // 3)] = t[: n // 3]
    return np.stack([dx * t + 11, dy * t - 7], axis=1).astype(np.int32)


def variants(kind, n, seed):
    rng = np.random.default_rng(seed)
    base = line(kind, n, seed)
    yield base
    off = base.copy()                         # a few points off the line: corners, inside, duplicates
    at = rng.choice(n, size=min(7, n), replace=False)
    off[at] += rng.integers(-1000, 1001, size=(len(at), 2)).astype(np.int32)
    off[at[-1]] = off[at[0]]
    yield off
    one = base.copy()                         # a single one, next to the line
    one[int(rng.integers(0, n))] += np.array([0, 1] if kind != "up" else [1, 0], np.int32)
    yield one
    ends = base.copy()                        # the first and the last row far out on both sides
    ends[0], ends[-1] = (ONE, -ONE), (-ONE, ONE)
    yield ends


@pytest.fixture(scope="module")
def ctx(hull_lib):
    with hull_lib.Context(0) as c:
        yield c


@pytest.mark.parametrize("kind", sorted(STEPS))
@pytest.mark.parametrize("n", [65536, 65537, 70001, 300001, 2000003])
def test_single(ctx, kind, n):
    for k, pts in enumerate(variants(kind, n + 1, n)):
        buf = torch.as_tensor(pts).cuda()
        for view in (buf[:-1], buf[1:]):       # an even and an odd first row
            assert ctx.compute(view).cpu().numpy().tolist() == oracle.hull(view.cpu().numpy()).tolist(), k


def test_two_lanes(hull_lib, ctx):
    sets = [p for kind in sorted(STEPS) for p in variants(kind, 66000, 5)]
    outs = [torch.empty(len(p), dtype=torch.int32, device="cuda") for p in sets]
    got = ctx.compute_multi([torch.as_tensor(p).cuda() for p in sets], outs)
    assert [h.cpu().numpy().tolist() for h in got] == [oracle.hull(p).tolist() for p in sets]


@pytest.mark.parametrize("n", [2, 1024, 1025, 2049, 5000, 16384, 16385, 16384 * 2 + 1, 50001, 400001])
def test_batched(ctx, n):
    parts = [p for kind in sorted(STEPS) for p in variants(kind, n, n + 1)]
    off = np.zeros(len(parts) + 1, np.int64)
    off[1:] = np.cumsum([len(p) for p in parts])
    v, o = (x.cpu().numpy() for x in ctx.compute_batched(torch.as_tensor(np.concatenate(parts)).cuda(),
                                                         torch.as_tensor(off).cuda()))
    for i, p in enumerate(parts):
        assert v[o[i]:o[i + 1]].tolist() == oracle.hull(p).tolist(), i


@pytest.mark.parametrize("n", [70001, 300001])
def test_out_of_range_on_the_line(hull_lib, ctx, n):
    """A coordinate beyond the limit is refused also where it lies on the line."""
    t = np.arange(n) - n // 2
    for at in (3, n // 2, n - 1):
        pts = np.stack([t * 4, t * 4], axis=1).astype(np.int32)
        pts[at] = (ONE + 4, ONE + 4)
        dev, off = torch.as_tensor(pts).cuda(), torch.tensor([0, n], device="cuda")
        for call in (lambda: ctx.compute(dev), lambda: ctx.compute_batched(dev, off)):
            with pytest.raises(hull_lib.HullError) as e:
                call()
            assert e.value.code == hull_lib.HULL_ERANGE


@pytest.mark.parametrize("n", [70001, 300001])
def test_capacity(hull_lib, ctx, n):
    pts = line("diagonal", n, 1)
    out = torch.full((1,), -3, dtype=torch.int32, device="cuda")
    with pytest.raises(hull_lib.HullError) as e:
        ctx.compute(torch.as_tensor(pts).cuda(), out=out)
    assert e.value.code == hull_lib.HULL_ECAPACITY and int(out[0]) == -3
    assert ctx.compute(torch.as_tensor(pts).cuda()).cpu().numpy().tolist() == oracle.hull(pts).tolist()

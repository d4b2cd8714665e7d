"""The star path (sample polygon, hull in angular order about an interior
point) at the edges of its kernels, every hull against the oracle: the
small-input kernel and its list sizes, the single-read front just above it,
the sectors for hulls of many vertices, the batched kernels' size classes,
and the inputs that it hands on."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1508_05931_gb300 import hull, workloads as W


@pytest.fixture(scope="module")
def ctx():
    with hull.Context(0) as c:
        yield c


def points(family, n, seed):
    rng = np.random.default_rng(seed)
    if family == "disk":
        return W.uniform_disk(n, 2.0 ** 29, seed)
    if family == "ring":
        return W.near_circle(n, 2.0 ** 28, seed)
    if family == "tiny_range":
        return rng.integers(-3, 4, size=(n, 2)).astype(np.int32)
    if family == "bytes":
        return np.clip(128 + 40 * rng.standard_normal((n, 2)), 0, 255).astype(np.int32)
    a = rng.standard_normal((n, 2)) * np.array([2.0 ** 26, 2.0 ** 26 / 300.0])
    c, s = np.cos(0.7), np.sin(0.7)
    return np.stack([c * a[:, 0] - s * a[:, 1], s * a[:, 0] + c * a[:, 1]], axis=1).astype(np.int32)


def check(ctx, pts):
    ref = oracle.hull(pts).tolist()
    t = torch.as_tensor(pts).cuda()
    assert ctx.compute(t).cpu().numpy().tolist() == ref
    if len(pts) <= hull.NOALLOC_MAX_POINTS:
        out = torch.empty(len(pts), dtype=torch.int32, device="cuda")
        h = hull.compute_noalloc(t, out)
        assert out[:h].cpu().numpy().tolist() == ref


# One block's limits: 64 points in one thread, 4,096 taken whole, 8,192 in the
# list (a ring of 16,500 leaves more, one of 16,000 fewer), 65,535 points;
# from 65,536 on the front, whose warps take chunks of 256 points.
@pytest.mark.parametrize("family", ["disk", "ring", "tiny_range", "bytes", "sliver"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 63, 64, 65, 1023, 4095, 4096, 4097, 16000, 16500, 65535, 65536, 65537,
                               65536 + 255, 150 * 16 * 256 + 1])
def test_sizes(ctx, family, n):
    check(ctx, points(family, n, n))


@pytest.mark.parametrize("distinct", [5, 40, 3000])
@pytest.mark.parametrize("n", [70001, 300000])
def test_duplicates_of_few(ctx, n, distinct):
    """Most raw survivors are duplicates of a candidate: the smallest index of
    every vertex, whichever copy came first."""
    rng = np.random.default_rng(distinct)
    check(ctx, W.uniform_disk(distinct, 2.0 ** 29, 3)[rng.integers(0, distinct, size=n)])


@pytest.mark.parametrize("n", [65536, 70001, 131071])
def test_odd_rows_and_repeated_calls(ctx, n):
    """Views that start on an odd row, twice each (the tables are left clear
    by a call that decides and not by one that does not)."""
    for family in ("disk", "ring", "disk"):
        buf = torch.as_tensor(points(family, n + 1, n)).cuda()
        for view in (buf[1:], buf[:-1], buf[1:]):
            assert ctx.compute(view).cpu().numpy().tolist() == oracle.hull(view.cpu().numpy()).tolist()


@pytest.mark.parametrize("n", [3, 100, 5000, 70000])
def test_degenerate_and_convex(ctx, n):
    t = np.arange(n) - n // 2
    y = (t.astype(np.int64) ** 2 * 4 // max(1, n)).astype(np.int64)
    for pts in (np.stack([t * 3, t * 5], 1), np.stack([t, 0 * t], 1), np.stack([0 * t, t], 1), np.full((n, 2), 9),
                np.stack([t, y], 1), np.stack([t, np.where(t == t[-1], 1, 0)], 1), np.repeat(np.stack([t, y], 1)[:: 7], 5, 0)):
        check(ctx, np.ascontiguousarray(pts.astype(np.int32)))


def test_range_and_capacity(ctx):
    for n in (100, 6000, 70000, 300000):
        pts = points("disk", n, 5)
        for at in (0, n // 2, n - 1):
            bad = pts.copy()
            bad[at] = ((1 << 29) + 1, 0)
            with pytest.raises(hull.HullError) as e:
                ctx.compute(torch.as_tensor(bad).cuda())
            assert e.value.code == hull.HULL_ERANGE
        out = torch.full((3,), -1, dtype=torch.int32, device="cuda")
        with pytest.raises(hull.HullError) as e:
            ctx.compute(torch.as_tensor(pts).cuda(), out=out)
        assert e.value.code == hull.HULL_ECAPACITY and (out.cpu().numpy() == -1).all()
        check(ctx, pts)


@pytest.mark.parametrize("families", [("disk",), ("sliver", "bytes", "disk"), ("ring", "tiny_range")])
def test_batched_size_classes(ctx, families):
    sizes = [0, 1, 2, 3, 64, 65, 1024, 1025, 1026, 2049, 16384, 16385, 16384 + 128 * 256, 32768, 32769, 50001]
    sets = [points(families[i % len(families)], n, 100 + i) if n else np.empty((0, 2), np.int32)
            for i, n in enumerate(sizes)]
    off = np.zeros(len(sizes) + 1, np.int64)
    off[1:] = np.cumsum(sizes)
    t = torch.as_tensor(np.concatenate(sets)).cuda()
    v, o = ctx.compute_batched(t, torch.as_tensor(off).cuda())
    v, o = v.cpu().numpy(), o.cpu().numpy()
    for i, p in enumerate(sets):
        ref = oracle.hull(p).tolist() if len(p) else []
        assert v[o[i]:o[i + 1]].tolist() == ref, (i, sizes[i])

"""The calls this library is used for, with their inputs, as measured cases.

A case names an entry point ("call"), a point family and a size; prepare()
builds the inputs on the GPU (or in pinned host memory for the host entry
point) and the context that a program keeps, run() makes one call.
"""
import math

import numpy as np
import torch

from paper_1508_05931_gb300 import hull, workloads

LIMIT = float(1 << 29)
FAMILIES = ("square", "disk", "gaussian", "aniso", "ellipse", "clusters", "ring", "bytes")
MLP_SHAPES = ((128, 64), (128,), (128, 128), (128,), (32, 128), (32,))

# Calls:
#   compute     hull.Context.compute on one device tensor
#   noalloc     hull.compute_noalloc on one device tensor (<= 65,536 points)
#   sliced      compute on rows 1.. of a larger device array (8-byte aligned only)
#   multi       compute_multi on several device tensors
#   host        compute_host_multi on pinned host tensors
#   batched     compute_batched, sizes log-uniform in [lo, hi], mixed families
#   proposal    compute_batched with the learned filter proposal
#   gradient    mlp_gradient: forward and backward of the proposal network


def listed():
    return [
        # One query's neighbourhood or one object's outline: the call's latency.
        {"name": "square_1k", "call": "compute", "family": "square", "n": 1000, "half": 1 << 20},
        # A caller that may not allocate (a plug-in, a pool's hook).
        {"name": "noalloc_20k", "call": "noalloc", "family": "gaussian", "n": 20011},
        # The everyday set: 100,000 points of a small coordinate range.
        {"name": "square_100k", "call": "compute", "family": "square", "n": 100000, "half": 1 << 20},
        # A shard of a larger array that starts at an odd row.
        {"name": "sliced_5m", "call": "sliced", "family": "disk", "n": 4999999},
        # Quantised data: pairs of 8-bit channels of a 4-megapixel image, full of duplicates.
        {"name": "bytes_4m", "call": "compute", "family": "bytes", "n": 4000000},
        # Half the points next to the hull: few are filtered, sort and chains dominate.
        {"name": "ring_4m", "call": "compute", "family": "ring", "n": 4000000},
        # Elongated data as it comes from projections and trajectories.
        {"name": "aniso_20m", "call": "compute", "family": "aniso", "n": 20000000, "ratio": 10.0},
        # The headline: the 20M square and the 20M disk in one call.
        {"name": "square_disk_20m", "call": "multi", "sets": "square:20000000 disk:20000000"},
        # The same from pinned host memory, copies included.
        {"name": "host_square_disk_20m", "call": "host", "sets": "square:20000000 disk:20000000"},
        # Thousands of hulls of uneven sizes in one call.
        {"name": "batch_4096", "call": "batched", "count": 4096, "lo": 1000, "hi": 1000000, "cap": 250000000},
        # A thousand alike anisotropic sets, with the learned proposal on.
        {"name": "batch_1024_proposal", "call": "proposal", "count": 1024, "lo": 19531, "hi": 19532,
         "cap": 21000000},
        # One mini-batch of the proposal network's training.
        {"name": "gradient_64", "call": "gradient", "rows": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["compute", "compute", "compute", "noalloc", "sliced", "multi", "host", "batched", "proposal",
                       "gradient"])
    if call == "compute":
        family = rng.choice(FAMILIES)
        case = {"call": call, "family": family,
                "n": _log_int(rng, 1000, 4000000 if family in ("ring", "bytes") else 20000000)}
    elif call == "noalloc":
        case = {"call": call, "family": rng.choice(FAMILIES), "n": _log_int(rng, 100, 65536)}
    elif call == "sliced":
        case = {"call": call, "family": rng.choice(("square", "disk", "gaussian", "aniso", "clusters")),
                "n": _log_int(rng, 1000, 20000000)}
    elif call in ("multi", "host"):
        k = rng.randint(2, 4)
        case = {"call": call, "sets": " ".join(
            "%s:%d" % (rng.choice(("square", "disk", "gaussian", "clusters")), _log_int(rng, 20000, 40000000 // k))
            for _ in range(k))}
    elif call == "batched":
        lo = _log_int(rng, 100, 10000)
        case = {"call": call, "count": _log_int(rng, 16, 4096), "lo": lo, "hi": _log_int(rng, 10 * lo, 1000000),
                "cap": 250000000}
    elif call == "proposal":
        lo = _log_int(rng, 1000, 20000)
        case = {"call": call, "count": _log_int(rng, 64, 1024), "lo": lo, "hi": _log_int(rng, lo + 1, 20 * lo),
                "cap": 40000000}
    else:
        case = {"call": call, "rows": _log_int(rng, 8, 1024)}
    if case.get("family") == "aniso":
        case["ratio"] = round(math.exp(rng.uniform(0.0, math.log(100.0))), 3)
    if case.get("family") == "square":
        case["half"] = 1 << rng.randint(16, 29)
    return case


def _sets(case):
    return [(f, int(n)) for f, n in (part.split(":") for part in case["sets"].split())]


def _polar(gen, n, dev):
    """Radius fractions (square roots of uniforms) and angles of n points."""
    r = torch.rand(n, generator=gen, device=dev, dtype=torch.float64).sqrt_()
    t = torch.rand(n, generator=gen, device=dev, dtype=torch.float64).mul_(2.0 * math.pi)
    return r, t


def _rounded(x, y):
    return torch.stack([x, y], dim=1).round_().clamp_(-LIMIT, LIMIT).to(torch.int32)


def _normal(gen, n, dev):
    return torch.randn((2, n), generator=gen, device=dev, dtype=torch.float64)


def _room(family, n):
    """Capacity for the vertices of a hull of n points: one point in eight
    where half of them lie on the circle, else 65,536 (a 20M disk has about
    a thousand)."""
    return max(1, min(n, max(n // 8, 65536) if family == "ring" else 65536))


def _points(family, n, gen, dev, half=1 << 29, ratio=10.0):
    """n points of a family, int32 (n, 2) on the device (the distributions
    of paper_1508_05931_gb300.workloads, drawn on the GPU)."""
    if family == "square":
        return torch.randint(-half, half, (n, 2), generator=gen, device=dev, dtype=torch.int32)
    if family == "bytes":
        # two correlated 8-bit channels
        a, b = _normal(gen, n, dev)
        x, y = 128.0 + 40.0 * a, 128.0 + 30.0 * a + 20.0 * b
        return _rounded(x.clamp_(0.0, 255.0), y.clamp_(0.0, 255.0))
    if family == "disk":
        r, t = _polar(gen, n, dev)
        return _rounded(LIMIT * r * torch.cos(t), LIMIT * r * torch.sin(t))
    if family == "ring":
        r, t = _polar(gen, n, dev)
        on = torch.rand(n, generator=gen, device=dev, dtype=torch.float64) < 0.5
        r = torch.where(on, torch.ones_like(r), r)
        return _rounded(0.5 * LIMIT * r * torch.cos(t), 0.5 * LIMIT * r * torch.sin(t))
    if family == "gaussian":
        a, b = _normal(gen, n, dev)
        return _rounded(2.0 ** 26 * a, 2.0 ** 26 * b)
    turn = float(torch.rand(1, generator=gen, device=dev)) * 2.0 * math.pi
    c, s = math.cos(turn), math.sin(turn)
    if family == "aniso":
        a, b = _normal(gen, n, dev)
        a, b = 2.0 ** 26 * a, (2.0 ** 26 / ratio) * b
        return _rounded(c * a - s * b, s * a + c * b)
    if family == "ellipse":
        r, t = _polar(gen, n, dev)
        a, b = 2.0 ** 28 * r * torch.cos(t), (2.0 ** 28 / ratio) * r * torch.sin(t)
        return _rounded(c * a - s * b, s * a + c * b)
    r, t = _polar(gen, 8, dev)
    sigma = 2.0 ** (20.0 + 5.0 * torch.rand(8, generator=gen, device=dev, dtype=torch.float64))
    which = torch.randint(0, 8, (n,), generator=gen, device=dev)
    a, b = _normal(gen, n, dev)
    return _rounded(2.0 ** 27 * (r * torch.cos(t))[which] + sigma[which] * a,
                    2.0 ** 27 * (r * torch.sin(t))[which] + sigma[which] * b)


def _batch(case, gen, dev, seed):
    """The batch's points and offsets.  batched: square, disk or Gaussian
    per instance; proposal: anisotropic Gaussian, elliptic disk or (as a
    stand-in for clusters) Gaussian, axis ratio log-uniform in [1, 100] and
    a rotation per instance."""
    count = case["count"]
    sizes = workloads.batch_sizes(count, seed, case["lo"], case["hi"], case["cap"])
    offsets = np.zeros(count + 1, dtype=np.int64)
    offsets[1:] = np.cumsum(sizes)
    pts = torch.empty((int(offsets[-1]), 2), dtype=torch.int32, device=dev)
    rng = np.random.default_rng(seed)
    family = torch.as_tensor(rng.integers(0, 3, size=count), device=dev)
    proposal = case["call"] == "proposal"
    ratio = torch.as_tensor(np.exp(rng.uniform(0.0, math.log(100.0), size=count)), device=dev)
    turn = torch.as_tensor(rng.uniform(0.0, 2.0 * math.pi, size=count), device=dev)
    size_d = torch.as_tensor(sizes, device=dev)
    step = max(1, count // 16)
    for b0 in range(0, count, step):
        b1 = min(count, b0 + step)
        lo, hi = int(offsets[b0]), int(offsets[b1])
        n = hi - lo
        inst = torch.repeat_interleave(torch.arange(b0, b1, device=dev), size_d[b0:b1], output_size=n)
        fam = family[inst]
        r, t = _polar(gen, n, dev)
        g = torch.sqrt(-2.0 * torch.log1p(-r * r))
        x, y = torch.cos(t), torch.sin(t)
        if proposal:
            rad = torch.where(fam == 1, 2.0 ** 28 * r, 2.0 ** 26 * g)
            a, b = rad * x, rad * y / torch.where(fam == 2, torch.ones_like(r), ratio[inst])
            c, s = torch.cos(turn[inst]), torch.sin(turn[inst])
            x, y = c * a - s * b, s * a + c * b
        else:
            sq = torch.rand((2, n), generator=gen, device=dev, dtype=torch.float64) * 2.0 - 1.0
            rad = torch.where(fam == 1, LIMIT * r, 2.0 ** 26 * g)
            x = torch.where(fam == 0, LIMIT * sq[0], rad * x)
            y = torch.where(fam == 0, LIMIT * sq[1], rad * y)
        pts[lo:hi] = _rounded(x, y)
    return pts, torch.as_tensor(offsets, device=dev)


def _params(seed):
    """Parameters of the proposal network (He-style, as training starts)."""
    rng = np.random.default_rng(seed)
    parts = [rng.standard_normal(s) * math.sqrt(2.0 / s[1]) if len(s) == 2 else 0.01 * rng.standard_normal(s)
             for s in MLP_SHAPES]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


def _rows(case, seed):
    """Feature rows (histogram shares and radii) and labels (discard
    fractions) in the ranges that the network is trained on."""
    rng = np.random.default_rng(seed)
    m = case["rows"]
    x = np.concatenate([rng.dirichlet(np.ones(32), size=m), rng.uniform(0.0, 1.0, size=(m, 32))], axis=1)
    return x.astype(np.float32), rng.uniform(0.0, 0.3, size=(m, 32)).astype(np.float32)


def prepare(case, seed):
    dev = torch.device("cuda", 0)
    call = case["call"]
    state = {"call": call}
    if call == "gradient":
        state["ctx"] = hull.Context(0)
        state["ctx"].mlp_set_params(_params(seed))
        state["x"], state["y"] = _rows(case, seed)
        return state
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    if call in ("batched", "proposal"):
        state["ctx"] = hull.Context(0, proposal=int(call == "proposal"))
        if call == "proposal":
            state["ctx"].mlp_set_params(_params(seed))
        state["pts"], state["offsets"] = _batch(case, gen, dev, seed)
        # room for the vertices: a few hundred per hull, zero where none are written
        state["out"] = torch.zeros(min(1024 * case["count"], state["pts"].shape[0]), dtype=torch.int32, device=dev)
        return state
    if call in ("multi", "host"):
        sets = [_points(f, n, gen, dev) for f, n in _sets(case)]
        if call == "host":
            state["sets"] = [torch.empty(t.shape, dtype=torch.int32, pin_memory=True).copy_(t) for t in sets]
        else:
            state["sets"] = sets
        state["outs"] = [torch.zeros(_room(f, n), dtype=torch.int32, device="cpu" if call == "host" else dev)
                         for f, n in _sets(case)]
        state["ctx"] = hull.Context(0)
        return state
    extra = 1 if call == "sliced" else 0
    pts = _points(case["family"], case["n"] + extra, gen, dev, case.get("half", 1 << 29), case.get("ratio", 10.0))
    state["pts"] = pts[extra:]
    state["out"] = torch.zeros(_room(case["family"], case["n"]), dtype=torch.int32, device=dev)
    if call != "noalloc":
        state["ctx"] = hull.Context(0)
    return state


def run(state):
    """One call.  Hulls come back as the caller's buffer (the vertices first)
    with their number."""
    call = state["call"]
    if call in ("compute", "sliced"):
        return [state["out"], len(state["ctx"].compute(state["pts"], out=state["out"]))]
    if call == "noalloc":
        return [state["out"], hull.compute_noalloc(state["pts"], state["out"])]
    if call == "multi":
        return [state["outs"], [len(h) for h in state["ctx"].compute_multi(state["sets"], state["outs"])]]
    if call == "host":
        return [state["outs"], [len(h) for h in state["ctx"].compute_host_multi(state["sets"], state["outs"])]]
    if call in ("batched", "proposal"):
        return list(state["ctx"].compute_batched(state["pts"], state["offsets"], out=state["out"]))
    g, loss = state["ctx"].mlp_gradient(state["x"], state["y"])
    return [g, np.float32(loss)]


def work(case):
    """Every point read once (8 bytes); the vertices are few beside them but
    on the ring, where about one point in twenty is one.  A hull compares
    integers: no floating-point work is counted."""
    call = case["call"]
    if call == "gradient":
        params = sum(int(np.prod(s)) for s in MLP_SHAPES)
        return {"bytes": 4 * (case["rows"] * 96 + 2 * params), "flops": 6 * case["rows"] * params}
    if call in ("multi", "host"):
        n = sum(k for _, k in _sets(case))
    elif call in ("batched", "proposal"):
        lo, hi = case["lo"], case["hi"]
        mean = (hi - lo) / math.log(hi / lo)
        n = int(min(case["cap"], case["count"] * mean))
    else:
        n = case["n"]
    return {"bytes": 8 * n + (n // 5 if case.get("family") == "ring" else 0), "flops": 0}


def exact(case, seed):
    """The gradient and the loss in float64 (on the FP16-rounded weights that
    the forward pass uses).  Hulls are vertex indices: whole numbers."""
    if case["call"] != "gradient":
        return None
    flat = _params(seed).astype(np.float16).astype(np.float64)
    p, at = [], 0
    for s in MLP_SHAPES:
        k = int(np.prod(s))
        p.append(flat[at:at + k].reshape(s))
        at += k
    w1, b1, w2, b2, w3, b3 = p
    x, y = (v.astype(np.float64) for v in _rows(case, seed))
    a1 = x @ w1.T + b1
    h1 = np.maximum(a1, 0.0)
    a2 = h1 @ w2.T + b2
    h2 = np.maximum(a2, 0.0)
    z = h2 @ w3.T + b3
    dz = 2.0 * (z - y) / z.size
    d2 = (dz @ w3) * (a2 > 0.0)
    d1 = (d2 @ w2) * (a1 > 0.0)
    grad = [d1.T @ x, d1.sum(0), d2.T @ h1, d2.sum(0), dz.T @ h2, dz.sum(0)]
    return [np.concatenate([g.ravel() for g in grad]), np.mean((z - y) ** 2)]

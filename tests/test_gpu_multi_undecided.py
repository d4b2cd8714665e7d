"""compute_multi with several inputs that the star path does not decide on one
lane: each goes on from its own points (a lane holds the raw survivors of one
input only), whatever stands before and behind it."""
import numpy as np
import pytest

import oracle
from paper_1508_05931_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N = 70000
SMALL = 20000                       # below the single-read front's 65,536 points


def points(kind, k):
    if kind == "ring":              # more vertices than one block takes: the sectors
        return W.near_circle(N + k, 2.0 ** 28, 10 + k)
    if kind == "line":              # no polygon: the paper's steps
        t = np.arange(N - 2 * k) - N // 2
        return np.stack([t * (3 + k), t * 5 - k], axis=1).astype(np.int32)
    if kind == "columns":           # two columns: no polygon with an interior, not on one line
        y = np.random.default_rng(30 + k).integers(-1 << 28, 1 << 28, size=N)
        return np.stack([np.arange(N) % 2 + k, y], axis=1).astype(np.int32)
    if kind == "small_ring":
        return W.near_circle(SMALL + k, 2.0 ** 27, 40 + k)
    if kind == "small":
        return W.uniform_disk(500 + k, 2.0 ** 27, 50 + k)
    return W.uniform_square(N + 3 * k, 1 << 28, 60 + k)


@pytest.mark.parametrize("proposal", [0, 1])
@pytest.mark.parametrize("kinds", [
    "ring square line", "line square ring", "line square line", "ring square ring", "ring ring ring", "columns square line",
    "line line", "ring line", "columns ring", "ring line line ring line", "ring square small", "line ring small_ring small",
    "small_ring line small_ring ring", "square square"])
def test_undecided_inputs_of_one_lane(hull_lib, kinds, proposal):
    sets = [points(kind, k) for k, kind in enumerate(kinds.split())]
    refs = [oracle.hull(p).tolist() for p in sets]
    dev = [torch.as_tensor(p).cuda() for p in sets]
    with hull_lib.Context(0, proposal=proposal) as c:
        if proposal:                # one lane: the learned proposal's buffers are per context
            c.mlp_set_params(np.zeros(int(hull_lib._lib.hull_mlp_num_params()), np.float32))
        for _ in range(2):
            outs = [torch.full((len(p),), -1, dtype=torch.int32, device="cuda") for p in sets]
            got = [h.cpu().numpy().tolist() for h in c.compute_multi(dev, outs)]
            assert got == refs

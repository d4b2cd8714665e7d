"""Stage times of calls that the star path's block hands on: the front's stages
are those of the pass that ran, not the empty marks of the next step."""
import numpy as np
import pytest

from paper_1508_05931_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N = 4_000_000
# 32 MB in no less than 3 us (10 TB/s); an empty slot between two events takes about 2.
LEAST_MS = 0.003


def columns():
    y = np.random.default_rng(4).integers(-1 << 28, 1 << 28, size=N)
    return np.stack([np.arange(N) % 2, y], axis=1).astype(np.int32)


@pytest.mark.parametrize("kind", ["disk", "ring", "columns"])
def test_front_stages_of_a_call(hull_lib, kind):
    pts = columns() if kind == "columns" else (W.near_circle if kind == "ring" else W.uniform_disk)(N, 2.0 ** 28, 3)
    t = torch.as_tensor(pts).cuda()
    with hull_lib.Context(0) as c:
        c.compute(t)
        c.set_profiling(True)
        c.compute(t)
        p = c.profile()
    assert p["calls"] == 1 and p["single_read_calls"] == 1 and p["raw_survivors"] > 0
    assert p["ms"]["polygon"] > LEAST_MS and p["ms"]["extremes"] > LEAST_MS

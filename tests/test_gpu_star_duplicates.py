"""Small inputs and batched instances made of few distinct points: copies of a
sector's candidate end before the list (smallest index of every vertex,
whichever copy the sample met), in one block's list and past its end."""
import numpy as np
import pytest

import oracle
from paper_1508_05931_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def copies(n, distinct, seed):
    rng = np.random.default_rng(seed)
    few = W.uniform_disk(distinct, 2.0 ** 29, seed) if seed % 2 else rng.integers(-4, 5, size=(distinct, 2)).astype(np.int32)
    return few[rng.integers(0, distinct, size=n)]


CASES = [(n, d) for n in (1025, 4097, 9000, 16384, 30000, 65535) for d in (2, 5, 40, 200, 1000)]


@pytest.mark.parametrize("n,distinct", CASES)
def test_single_and_noalloc(hull_lib, n, distinct):
    with hull_lib.Context(0) as c:
        for seed in (1, 2, 3, 4):
            pts = copies(n, distinct, seed)
            ref = oracle.hull(pts).tolist()
            t = torch.as_tensor(pts).cuda()
            assert c.compute(t).cpu().numpy().tolist() == ref
            out = torch.empty(n, dtype=torch.int32, device="cuda")
            assert out[:hull_lib.compute_noalloc(t, out)].cpu().numpy().tolist() == ref


def test_batched(hull_lib):
    parts = [copies(n, d, s) for n, d in CASES for s in (1, 2)]
    off = np.zeros(len(parts) + 1, np.int64)
    off[1:] = np.cumsum([len(p) for p in parts])
    with hull_lib.Context(0) as c:
        v, o = (x.cpu().numpy() for x in c.compute_batched(torch.as_tensor(np.concatenate(parts)).cuda(),
                                                             torch.as_tensor(off).cuda()))
    for i, p in enumerate(parts):
        assert v[o[i]:o[i + 1]].tolist() == oracle.hull(p).tolist(), i

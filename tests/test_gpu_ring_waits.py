"""The bulk-copy rings of the single-read pass and of the batched pass with a
spin limit of one iteration: a warp whose next chunk is not there at once gives
up, the call reports HULL_ETIMEOUT (never a hull of the points that it has
seen), nothing hangs, and the next call with the normal limit is exact."""
import numpy as np
import pytest

import oracle
from paper_1508_05931_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def outcomes(hull_lib, call, ref):
    codes = []
    for _ in range(5):
        try:
            assert call() == ref
            codes.append(hull_lib.HULL_OK)
        except hull_lib.HullError as e:
            codes.append(e.code)
    return codes


def test_single_read_pass(hull_lib):
    pts = W.uniform_disk(4_000_000, 2.0 ** 28, 3)
    ref = oracle.hull(pts).tolist()
    t = torch.as_tensor(pts).cuda()
    with hull_lib.Context(0, spin_limit=1) as c:
        codes = outcomes(hull_lib, lambda: c.compute(t).cpu().numpy().tolist(), ref)
    assert set(codes) <= {hull_lib.HULL_OK, hull_lib.HULL_ETIMEOUT} and hull_lib.HULL_ETIMEOUT in codes
    with hull_lib.Context(0) as c:
        assert c.compute(t).cpu().numpy().tolist() == ref


def test_batched_pass_with_an_undecided_instance(hull_lib):
    """The instances that the pass does not decide go on to the general path
    only when the pass itself was whole."""
    parts = [W.uniform_disk(300_000, 2.0 ** 28, i) for i in range(40)] + [W.near_circle(30_000, 2.0 ** 28, 5)]
    refs = [oracle.hull(p).tolist() for p in parts]
    off = np.zeros(len(parts) + 1, np.int64)
    off[1:] = np.cumsum([len(p) for p in parts])
    t, o = torch.as_tensor(np.concatenate(parts)).cuda(), torch.as_tensor(off).cuda()

    def call(c):
        v, oo = (x.cpu().numpy() for x in c.compute_batched(t, o))
        return [v[oo[i]:oo[i + 1]].tolist() for i in range(len(parts))]

    with hull_lib.Context(0, spin_limit=1) as c:
        codes = outcomes(hull_lib, lambda: call(c), refs)
    assert set(codes) <= {hull_lib.HULL_OK, hull_lib.HULL_ETIMEOUT} and hull_lib.HULL_ETIMEOUT in codes
    with hull_lib.Context(0) as c:
        assert call(c) == refs

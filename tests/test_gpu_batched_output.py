"""What a batched call that fails leaves behind when some instances go on to the
general path: the output buffer untouched, the offsets of all hulls."""
import numpy as np
import pytest

import oracle
from paper_1508_05931_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("order", [1, -1])
@pytest.mark.parametrize("ring", [6000, 30000])
def test_capacity_with_undecided_instances(hull_lib, ring, order):
    parts = [W.uniform_disk(5000, 2.0 ** 28, 1), W.near_circle(ring, 2.0 ** 28, 2), W.uniform_square(20000, 1 << 28, 3)][::order]
    refs = [oracle.hull(p).tolist() for p in parts]
    off = np.zeros(len(parts) + 1, np.int64)
    off[1:] = np.cumsum([len(p) for p in parts])
    t, o = torch.as_tensor(np.concatenate(parts)).cuda(), torch.as_tensor(off).cuda()
    total = sum(map(len, refs))
    oo = torch.empty(len(parts) + 1, dtype=torch.int64, device="cuda")
    with hull_lib.Context(0) as c:
        for cap in (total - 1, total - len(refs[-1]), total):
            out = torch.full((total,), -7, dtype=torch.int32, device="cuda")
            code = hull_lib._lib.hull_compute_batched(c.handle, t.data_ptr(), o.data_ptr(), len(parts), out.data_ptr(), cap,
                                                      oo.data_ptr(), torch.cuda.current_stream().cuda_stream)
            assert oo.cpu().numpy().tolist() == np.cumsum([0] + [len(r) for r in refs]).tolist()
            if cap < total:
                assert code == hull_lib.HULL_ECAPACITY and (out == -7).all()
            else:
                assert code == hull_lib.HULL_OK and out.cpu().numpy().tolist() == sum(refs, [])


def test_range_with_undecided_instances(hull_lib):
    bad = W.uniform_square(20000, 1 << 28, 3).copy()
    bad[777] = [0, (1 << 29) + 1]
    parts = [W.uniform_disk(5000, 2.0 ** 28, 1), W.near_circle(30000, 2.0 ** 28, 2), bad]
    off = np.zeros(len(parts) + 1, np.int64)
    off[1:] = np.cumsum([len(p) for p in parts])
    out = torch.full((int(off[-1]),), -7, dtype=torch.int32, device="cuda")
    with hull_lib.Context(0) as c, pytest.raises(hull_lib.HullError) as e:
        c.compute_batched(torch.as_tensor(np.concatenate(parts)).cuda(), torch.as_tensor(off).cuda(), out=out)
    assert e.value.code == hull_lib.HULL_ERANGE and (out == -7).all()


def test_misaligned_points_are_refused(hull_lib):
    """Points are read eight bytes at a time: a pointer between two of them is
    an error before any launch, as in the single-hull calls."""
    flat = torch.zeros(2 * 300 + 1, dtype=torch.int32, device="cuda")
    off = torch.tensor([0, 100, 300], device="cuda")
    with hull_lib.Context(0) as c:
        with pytest.raises(hull_lib.HullError) as e:
            c.compute_batched(flat[1:].view(300, 2), off)
        assert e.value.code == hull_lib.HULL_EINVAL
        v, o = c.compute_batched(flat[:-1].view(300, 2), off)
        assert o.cpu().numpy().tolist() == [0, 1, 2] and v[:2].cpu().numpy().tolist() == [0, 0]

"""The batched call's general path (one block per instance, or the segmented
passes) on every instance: a context whose caller sets the boundary between
the two (hull_config.batched_seg_min) does not take the star path."""
import re

import numpy as np
import pytest

from paper_1508_05931_gb300 import learned as L, workloads as W
from test_gpu_batched import check, mixed_parts, run_batch, sort_path_parts

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("seg_min", [65536, 1 << 30])
def test_a_set_boundary_is_the_general_path(hull_lib, seg_min):
    """With a spin limit of one the star path's copy rings time out on these
    instances; the general path has no such wait."""
    parts = [W.uniform_disk(300_000, 2.0 ** 28, i) for i in range(40)]
    with hull_lib.Context(0, spin_limit=1, batched_seg_min=seg_min) as c:
        check(parts, *run_batch(c, parts))


@pytest.mark.parametrize("seg_min", [65536, 1 << 30])
def test_learned_proposal_on_every_large_instance(hull_lib, seg_min):
    from oracle import mlp as OM
    parts = [L.instance(k, 300_000, 400 + k) for k in range(3)] + [L.instance(k, 262_143 + k, 410 + k) for k in range(2)]
    parts += mixed_parts(5)
    with hull_lib.Context(0, proposal=1, batched_seg_min=seg_min) as c:
        for params in (OM.init_params(11), np.zeros(OM.N_PARAMS, np.float32)):
            c.mlp_set_params(params)
            check(parts, *run_batch(c, parts))


@pytest.mark.parametrize("block", [256, 512])
def test_sort_paths_both_block_sizes(hull_lib, tmp_path, monkeypatch, block):
    cache = tmp_path / "tune.json"
    monkeypatch.setenv("GBHULL_AUTOTUNE_CACHE", str(cache))
    parts = sort_path_parts() + mixed_parts(6)
    with hull_lib.Context(0, autotune=True) as c:        # writes the cache for this device
        run_batch(c, parts)
    cache.write_text(re.sub(r'(batched_(?:small|large|seg_block)": )\d+', r"\g<1>%d" % block, cache.read_text()))
    for seg_min in (16385, 1 << 30):
        with hull_lib.Context(0, autotune=True, batched_seg_min=seg_min) as c:
            check(parts, *run_batch(c, parts))

"""The tuner picks one of its shapes also for a batch that is stepped by one-tile
blocks (for when the batch grows), and leaves the members as they were.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

SHAPES = {(t, s, l) for t in (64, 128) for s in (8, 16) for l in (16, 32)}


@pytest.mark.parametrize("nx,ny", [(96, 70), (1500, 1000)])  # one-tile blocks, the persistent kernel
def test_tuned_shape_is_a_candidate(nx, ny):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09534_gb300 import build
    build.build()
    import paper_1710_09534_gb300 as T
    w = W.random_lattice(nx, ny, 9, edges=(0, 0, 1, 3), lid_u=0.01)
    alone, member = (T.lattice_from_workload(w, "fp32") for _ in range(2))
    batch = T.Batch("fp32", 1, 2 * T.Batch.tiles_needed(nx, ny), member.wall_nodes())
    batch.config(threads=64, rows_small=5, rows_large=7)
    batch.add(member)
    batch.step(3)
    cfg = batch.tune(trial_steps=3)
    assert (cfg["threads"], cfg["rows_small"], cfg["rows_large"]) in SHAPES
    assert cfg["ms_per_step"] > 0
    batch.step(4)
    batch.synchronize()
    alone.step(7)
    assert np.array_equal(alone.state(), member.state())

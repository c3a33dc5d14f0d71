"""A batch's capacity is that of its configured shape: what a shape fits is stepped
also where the one-tile blocks of a small batch would need more items, and what it
does not fit is refused also where they would need fewer.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09534_gb300 import build
    build.build()
    import paper_1710_09534_gb300 as T
    return T


def lattices(T):
    ws = [W.random_lattice(250, 130, 7 + i, edges=(0, 0, 1, 2)) for i in range(2)]
    return [T.lattice_from_workload(w, "fp32") for w in ws], [T.lattice_from_workload(w, "fp32") for w in ws]


@pytest.mark.parametrize("rows,fits", [(32, 2 * 3 * 5), (2, 2 * 3 * 65)])  # strips of 124 columns, segments of `rows`
def test_capacity_of_the_configured_shape(T, rows, fits):
    alone, members = lattices(T)
    walls = sum(L.wall_nodes() for L in members)
    for cap in (fits, fits - 1):
        batch = T.Batch("fp32", 2, cap, walls)
        batch.config(threads=128, rows_small=rows, rows_large=rows)
        for L in members:
            batch.add(L)
        if cap < fits:
            with pytest.raises(T.TlbError) as e:
                batch.step(3)
            assert e.value.code == T.ENOMEM
        else:
            batch.step(3)
            batch.synchronize()
            for a, m in zip(alone, members):
                a.step(3)
                assert np.array_equal(a.state(), m.state())
        for L in members:
            batch.remove(L)
        batch.close()

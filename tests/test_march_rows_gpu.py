"""Lattices of less than one wave of marching blocks, whose segments get a length
of 4 to 15 rows (rows_for), at ragged sizes: stepped alone they take k_step_march,
as members of a batch of this size one-tile blocks, and the raw states must be
equal bit for bit.  So must those of a lattice of the 16-bit MRT collision beyond
its tile limit and of a large batch that holds it.
"""
import numpy as np
import pytest

from test_tile_gpu import T, batch_of, workload  # noqa: F401  (T is the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,nx,ny,mrt", [
    ("fp32", 601, 600, False), ("fp32", 1003, 351, False), ("fp32", 125, 2801, False), ("fp32", 777, 777, True),
    ("fp16", 500, 613, False), ("fp16", 2048, 151, False), ("bf16", 860, 811, False), ("fp16", 1500, 1471, True)])
@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("edges", [(0, 0, 1, 3), (1, 2, 0, 0)])
def test_march_alone_equals_the_batch_member(T, precision, nx, ny, mrt, uniform, edges):  # noqa: F811
    w = workload(nx, ny, edges, ("disc",), mrt, uniform, seed=12)
    alone = T.lattice_from_workload(w, precision)
    batch, (member,) = batch_of(T, precision, [w])
    for n in (4, 3):
        alone.step(n)
        batch.step(n)
    batch.synchronize()
    ref = alone.state()
    assert np.isfinite(ref).all()
    assert np.array_equal(ref, member.state())

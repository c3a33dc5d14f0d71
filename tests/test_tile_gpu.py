"""The one-launch step of small lattices (k_step_tile) at the edges of its tiles.

Stepped alone, lattices of these sizes take k_step_tile.  As members of a batch
that also holds a large lattice they take the marching items and near-wall tiles
of k_batch_interior, and the large lattice stepped alone takes k_step_march.  All run the same arithmetic, so the raw states must be equal
bit for bit, for every storage, collision model, edge kind and ragged size; so
must those of a batch of small lattices only (k_batch_tile).  In FP64 the state
also equals the oracle within the parity bound.
"""
import numpy as np
import pytest

import workloads as W
from oracle import OracleLattice

from test_parity_gpu import assert_parity

pytestmark = pytest.mark.gpu

# one tile (32 x 8, 32 x 4) and its remainders, the smallest lattices, lid rows
# that open a tile (ny % 8 == 1, ny % 4 == 1), every edge kind
SHAPES = [
    (3, 3, (0, 0, 0, 0), ()),
    (3, 6, (1, 2, 2, 3), ()),
    (31, 9, (0, 0, 1, 3), ("pillar",)),
    (32, 8, (0, 0, 1, 2), ()),
    (33, 17, (1, 2, 2, 3), ("pillar",)),
    (64, 16, (0, 0, 0, 0), ("disc",)),
    (65, 33, (0, 0, 2, 3), ("corner", "disc")),
    (97, 41, (2, 1, 1, 1), ("corner", "pillar")),
    (130, 70, (0, 0, 1, 2), ("disc", "corner")),
]


@pytest.fixture(scope="module")
def T():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09534_gb300 import build
    build.build()
    import paper_1710_09534_gb300 as T
    return T


# a size that takes the marching kernel, per storage
LARGE = {"fp64": (1800, 1670), "fp32": (1250, 1130), "fp16": (900, 840), "bf16": (900, 840)}


def workload(nx, ny, edges, solids, mrt, uniform, seed=5):
    w = W.random_lattice(nx, ny, seed, edges=edges, solids=solids, lid_u=0.01 if edges[3] == 3 else 0.0)
    if uniform:
        w.params.update(rho1=1.0, rho2=1.0, rho3=1.0, nu1=0.1, nu2=0.1, nu3=0.1)
    if mrt:
        w.params.update(collision=1.0, mrt_s_f=1.3, mrt_s_g=1.2)
    return w


def batch_of(T, precision, ws):
    lats = [T.lattice_from_workload(w, precision) for w in ws]
    batch = T.Batch(precision, len(ws), sum(T.Batch.tiles_needed(w.nx, w.ny) for w in ws),
                    sum(max(1, L.wall_nodes()) for L in lats))
    for L in lats:
        batch.add(L)
    return batch, lats


@pytest.mark.parametrize("threads", [64, 128])
@pytest.mark.parametrize("precision,mrt,uniform", [
    ("fp64", False, True), ("fp64", False, False), ("fp64", True, True), ("fp32", False, True), ("fp32", False, False),
    ("fp32", True, False), ("fp16", False, True), ("fp16", True, True), ("bf16", False, False)])
def test_alone_equals_batch_members(T, precision, mrt, uniform, threads):
    ws = [workload(*s, mrt, uniform) for s in SHAPES]
    large = workload(*LARGE[precision], (0, 0, 1, 3), ("disc",), mrt, uniform)
    alone = [T.lattice_from_workload(w, precision) for w in ws + [large]]
    small, sm = batch_of(T, precision, ws)
    mixed, mx = batch_of(T, precision, ws + [large])
    mixed.config(threads=threads, rows_small=8, rows_large=32)
    for n in (4, 3):
        for L in alone:
            L.step(n)
        small.step(n)
        mixed.step(n)
    small.synchronize()
    mixed.synchronize()
    for i, (w, a) in enumerate(zip(ws + [large], alone)):
        ref = a.state()
        assert np.isfinite(ref).all()
        assert np.array_equal(ref, mx[i].state()), w.name
        if i < len(ws):
            assert np.array_equal(ref, sm[i].state()), w.name


@pytest.mark.parametrize("nx,ny,edges,solids", [s for s in SHAPES if s[0] > 16])
@pytest.mark.parametrize("uniform", [True, False])
def test_fp64_equals_the_oracle(T, nx, ny, edges, solids, uniform):
    w = workload(nx, ny, edges, solids, False, uniform, seed=8)
    L = T.lattice_from_workload(w, "fp64")
    O = OracleLattice(w.nx, w.ny, w.edges, w.mask, w.params)
    O.set_fields(w.c1, w.c2, w.ux, w.uy, w.p)
    O.param_dict = dict(w.params)
    L.step(40)
    O.step(40)
    assert_parity(L, O, what=w.name)

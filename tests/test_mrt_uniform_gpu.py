"""A uniform state at rest is a fixed point of the MRT update: the collision conserves
sum_k f^i_k (Eq. 1a) and nothing streams in or out of balance, so c may not drift in
FP64, whatever the rounding of the rates.  The bound is one rounding of c for the
whole run (the populations settle in the first steps).
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("inplace", [False, True])
@pytest.mark.parametrize("c1,c2", [(0.3, 0.2), (0.61, 0.17), (0.05, 0.9)])
@pytest.mark.parametrize("s_f", [0.7, 1.1, 1.2, 1.3, 1.7])
def test_uniform_state_does_not_drift(s_f, c1, c2, inplace):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09534_gb300 import build
    build.build()
    import paper_1710_09534_gb300 as T
    p = W.params()
    p.update(collision=1.0, mrt_s_f=s_f, mrt_s_g=1.3)
    L = T.Lattice(40, 30, "fp64", (0, 0, 0, 0), inplace=inplace)
    L.set_geometry(None)
    L.set_params(p)
    one = np.ones((30, 40))
    L.set_fields(c1 * one, c2 * one, 0 * one, 0 * one)
    L.step(2000)
    f = L.fields(("c1", "c2"))
    assert np.abs(f["c1"] - c1).max() <= np.spacing(c1)
    assert np.abs(f["c2"] - c2).max() <= np.spacing(c2)

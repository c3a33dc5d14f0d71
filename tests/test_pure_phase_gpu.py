"""A pure phase has no chemical potential: c (1 - c)(1 - 2c) and the Laplacian vanish
exactly at c = 0 and c = 1, whatever the rounding of the parameters (Eq. 8).  Read from
the initial state, in which c has those values exactly.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [1e-3, 7e-4, 3.3e-3, 1.7e-2])
@pytest.mark.parametrize("c1,c2", [(1.0, 0.0), (0.0, 1.0), (0.0, 0.0)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dims", [2, 3])
def test_mu_of_a_pure_phase_is_zero(dims, sigma, c1, c2, precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09534_gb300 import build
    build.build()
    import paper_1710_09534_gb300 as T
    shape = (6, 8) if dims == 2 else (5, 6, 8)
    L = T.Lattice(8, 6, precision, (0,) * 4) if dims == 2 else T.Lattice3D(8, 6, 5, (0,) * 6, precision=precision)
    L.set_geometry(None)
    L.set_params(W.params(sigma=(sigma,) * 3))
    one = np.ones(shape)
    L.set_fields(c1 * one, c2 * one, *[0 * one] * dims)
    f = L.fields(("mu1", "mu2", "mu3"))
    assert all((f[k] == 0).all() for k in f)

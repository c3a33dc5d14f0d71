"""The FP32 D3Q19 update over padded rows (k3_update_wide, 16-byte copies into the
block's stage) where its blocks and rows end: widths around a multiple of 32, a
plane that is not a multiple of a block, the smallest lattice; both updates,
against the oracle within the FP32 bounds.
"""
import pytest

import workloads as W

from test_d3q19_gpu import T, fp32_errors, pair  # noqa: F401  (T is the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("shape,edges,solids", [
    ((3, 3, 3), (0, 0, 0, 0, 0, 0), ()),
    ((31, 9, 7), (0, 0, 1, 2, 0, 0), ()),
    ((32, 9, 7), (1, 2, 0, 0, 2, 1), ("pillar",)),
    ((33, 13, 11), (0, 0, 1, 2, 0, 0), ("sphere",)),
    ((95, 10, 9), (2, 1, 1, 1, 0, 0), ("corner",)),      # rows padded by one element
    ((160, 8, 5), (0, 0, 2, 1, 1, 2), ()),
])
def test_wide_update_within_fp32_bounds_of_the_oracle(T, shape, edges, solids, uniform):  # noqa: F811
    w = W.random_lattice3(*shape, 41, edges=edges, solids=solids)
    if uniform:
        w.params.update(rho1=1.0, rho2=1.0, rho3=1.0, nu1=0.1, nu2=0.1, nu3=0.1)
    L, O = pair(T, w, "fp32")
    L.step(30)
    O.step(30)
    bad = {k: v for k, v in fp32_errors(L.fields(), O.fields()).items() if not v[0] < v[1]}
    assert not bad, f"{w.name}: {bad}"

"""tlb_profile_read: a two-buffer lattice steps by one launch, so the near-wall kernel
has neither launches nor time; an in-place one with walls has both.
"""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(130, 70), (1250, 1130)])
@pytest.mark.parametrize("inplace", [False, True])
def test_near_wall_time_is_that_of_its_launches(nx, ny, inplace):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09534_gb300 import build
    build.build()
    import paper_1710_09534_gb300 as T
    w = W.random_lattice(nx, ny, 6, edges=(0, 0, 1, 2))
    L = T.lattice_from_workload(w, "fp32", inplace=inplace)
    L.step(2)
    L.profile(True)
    L.step(6)
    interior_ms, wall_ms, interior_n, wall_n = L.profile_read()
    assert interior_n == 6 and interior_ms > 0
    assert (wall_n, wall_ms > 0) == ((6, True) if inplace else (0, False))
    if not inplace:
        assert wall_ms == 0

"""Read-out into host memory that is in use: the buffer of tlb_read_fields and
tlb3_read_fields is written by copies in stream order and by nothing before them.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1710_09534_gb300", "csrc")
NAMES = ("c1", "c2", "ux", "uy", "p")


def test_mapping_the_pages_keeps_the_contents(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    src, lib = tmp_path / "m.cpp", tmp_path / "m.so"
    src.write_text('#include "tlbm_host.h"\n'
                   'extern "C" int map_pages(void* p, size_t n) { return tlb::map_host_pages(p, n); }\n')
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    f = ctypes.CDLL(str(lib)).map_pages
    f.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
    a = np.random.default_rng(3).integers(1, 256, 300_000).astype(np.uint8)
    want = a.copy()
    for at, n in ((0, a.size), (1, a.size - 1), (4095, 4097), (77, 1), (5, 0)):
        f(a.ctypes.data + at, n)  # (whether the kernel knows the call is another matter)
        assert np.array_equal(a, want), (at, n)
    f(None, 4096)  # not mapped: refused, not a fault


@pytest.fixture(scope="module")
def T():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09534_gb300 import build
    build.build()
    import paper_1710_09534_gb300 as T
    return T


def make(T, dims):
    if dims == 2:
        w = W.random_lattice(512, 512, 23, edges=(0, 0, 1, 2))
        return T.lattice_from_workload(w, "fp64"), T.FIELDS
    w = W.random_lattice3(64, 48, 48, 23, edges=(0, 0, 1, 2, 0, 0))
    return T.lattice3_from_workload(w), T.FIELDS3


def read_into(T, L, dims, mask, out):
    f = T.load_library().tlb_read_fields if dims == 2 else T.load_library().tlb3_read_fields
    return f(L._h, mask, out.ctypes.data_as(ctypes.POINTER(ctypes.c_double)))


@pytest.mark.gpu
@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("dims", [2, 3])
def test_queued_upload_from_the_buffer_keeps_its_values(T, dims, pinned):
    import torch
    L, fields = make(T, dims)
    n, mask = len(NAMES), sum(1 << fields.index(k) for k in NAMES)
    host = torch.randn(n * L.n, dtype=torch.float64)
    host = host.pin_memory() if pinned else host
    want, dev = host.clone(), torch.zeros(n * L.n, dtype=torch.float64, device="cuda")
    L.step(1500)  # keeps the stream busy while the upload waits its turn
    dev.copy_(host, non_blocking=True)
    assert read_into(T, L, dims, mask, host.numpy()) == 0
    torch.cuda.synchronize()
    assert torch.equal(dev.cpu(), want)
    ref = np.empty(n * L.n)
    assert read_into(T, L, dims, mask, ref) == 0
    assert np.array_equal(host.numpy(), ref) and np.isfinite(ref).all()


@pytest.mark.gpu
def test_new_fields_from_the_staging_buffer_that_receives_the_next_ones(T):
    import torch
    A, _ = make(T, 2)
    B, _ = make(T, 2)
    first = A.fields(NAMES)
    stage = torch.from_numpy(np.stack([first[k] for k in NAMES])).pin_memory()
    up = torch.empty_like(stage, device="cuda")
    A.step(1500)
    up.copy_(stage, non_blocking=True)
    A.set_fields_device(up[0], up[1], up[2], up[3], up[4])
    A.step(3)
    got = A.fields(NAMES, out=stage.numpy())
    B.set_fields(*(first[k] for k in NAMES))
    B.step(3)
    want = B.fields(NAMES)
    assert all(np.array_equal(got[k], want[k]) for k in NAMES)


@pytest.mark.gpu
@pytest.mark.parametrize("dims", [2, 3])
def test_refused_readout_leaves_the_buffer(T, dims):
    L, _ = make(T, dims)
    out = np.full(16, 7.0)
    for mask in (0, 1 << 20):
        assert read_into(T, L, dims, mask, out) < 0
    assert (out == 7.0).all()

"""Kernels launched as dependent launches (launch_dependent) are resident while
the launch before them still writes the state they read, and wait for it by
griddepcontrol.wait.  That orders plain loads only: what a step writes must not
be read through the read-only path, nor through a __restrict__ kernel argument,
whose loads the compiler may move above the wait.
"""
import os
import re

import numpy as np
import pytest

import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1710_09534_gb300", "csrc")
# written by the host or by an ordinary launch only
CONSTANT = {"cls", "walls", "items", "descs", "kind", "lnk"}
SOURCES = {f: re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
           for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}


def dependent_kernels():
    names = set()
    for text in SOURCES.values():
        names |= set(re.findall(r"launch_dependent\(&(?:tlb3::)?(k\w+)", text))
        for m in re.finditer(r"launch_dependent\(k,", text):  # auto* k = cond ? &k_a : &k_b;
            at = text.rindex("auto* k =", 0, m.start())
            names |= set(re.findall(r"&(?:tlb3::)?(k\w+)", text[at:text.index(";", at)]))
    return names


def body(text, at):
    """The parameters of the function whose name is at `at`, and its body."""
    depth, i = 0, text.index("(", at)
    start = i
    while True:
        depth += {"(": 1, ")": -1}.get(text[i], 0)
        i += 1
        if depth == 0:
            break
    params, j = text[start + 1:i - 1], text.index("{", i)
    start, depth = j, 0
    while True:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
        if depth == 0:
            return params, text[start:j]


def definition(name):
    for text in SOURCES.values():
        m = re.search(r"(?:__global__|__device__)[^;{}()]*?(?:__launch_bounds__\([^{};]*?\)\s*)?\b" + name + r"\(", text)
        if m:
            return body(text, m.end() - 1)
    raise AssertionError(f"{name} not found")


def test_dependent_kernels_read_the_state_by_plain_loads():
    kernels = dependent_kernels()
    assert {"k_step_tile", "k_step_march", "k_batch_interior", "k_batch_tile", "k3_csum", "k3_mu", "k3_update",
            "k3_update_wide"} <= kernels
    for k in kernels:
        for p in definition(k)[0].split(","):
            if "__restrict__" in p:
                assert p.split()[-1] in CONSTANT, f"{k}: {p.strip()}"
    for f in sorted(kernels | {"interior_tile", "tile_step", "wall_tile", "node3", "pair3", "update3_node"}):
        code = definition(f)[1]
        assert "__ldg" not in code and "ld_any<true>" not in code, f
        # the accessors of the populations default to the read-only path
        for call in re.findall(r"\b(?:ld_pop|ld_lo|ld_pair|order_params)<([^>(]*)", code):
            assert call.split(",")[1:2] == [" false"], f"{f}: <{call}>"


@pytest.fixture(scope="module")
def T():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09534_gb300 import build
    build.build()
    import paper_1710_09534_gb300 as T
    return T


@pytest.mark.gpu
@pytest.mark.parametrize("precision,nx,ny", [
    ("fp64", 130, 70), ("fp32", 257, 129), ("fp16", 257, 129), ("bf16", 130, 70),
    ("fp64", 1800, 1670), ("fp32", 1250, 1130), ("fp16", 900, 840), ("bf16", 900, 840)])
@pytest.mark.parametrize("uniform", [True, False])
def test_overlapping_steps_equal_steps_one_at_a_time(T, precision, nx, ny, uniform):
    w = W.random_lattice(nx, ny, 17, edges=(0, 0, 1, 3), solids=("disc",), lid_u=0.01)
    if uniform:
        w.params.update(rho1=1.0, rho2=1.0, rho3=1.0, nu1=0.1, nu2=0.1, nu3=0.1)
    A, B = (T.lattice_from_workload(w, precision) for _ in range(2))
    A.step(40)
    for _ in range(40):
        B.step(1)
        B.sync()
    assert np.array_equal(A.state(), B.state())


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("uniform", [True, False])
def test_overlapping_steps_equal_steps_one_at_a_time_d3q19(T, precision, uniform):
    w = W.random_lattice3(96, 40, 48, 17, edges=(0, 0, 1, 2, 0, 0), solids=("sphere",))
    if uniform:
        w.params.update(rho1=1.0, rho2=1.0, rho3=1.0, nu1=0.1, nu2=0.1, nu3=0.1)
    A, B = (T.lattice3_from_workload(w, precision=precision) for _ in range(2))
    A.step(40)
    for _ in range(40):
        B.step(1)
        B.sync()
    assert np.array_equal(A.state(), B.state())

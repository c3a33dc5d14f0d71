"""The stored DRAM traffic is keyed by the sources of the kernel it was captured from:
the file that defines that kernel is among them, and the capture names it.
"""
import json
import os
import re

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1710_09534_gb300", "csrc")


def test_the_timed_kernels_file_is_in_the_key():
    kernels = {k.split("<")[0] for k in bench.KERNEL.values()}
    defined = {k: [f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))
                   and re.search(r"\n" + k + r"\(const ", open(os.path.join(CSRC, f)).read())] for k in kernels}
    with open(os.path.join(ROOT, "profiles", "interior_traffic.json")) as f:
        about = json.load(f)["about"]
    for k, files in defined.items():
        assert files and set(files) <= set(bench.INTERIOR_SOURCES), (k, files)
        assert k in about

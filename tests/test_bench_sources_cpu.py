"""The bench reports a kernel's DRAM traffic only while the record's hash is
that of the kernel's sources: the hash covers every file of device code that
the kernel's unit includes (the checks of the debug build, which the release
library compiles to nothing, and the host's declarations aside)."""
import os
import re

import bench

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_17770_gb300", "csrc")


def _device_sources(name, seen):
    if name in seen or name == "ctf_debug.cuh" or not name.endswith((".cu", ".cuh")):
        return seen
    seen.add(name)
    for inc in re.findall(r'#include "([^"]+)"', open(os.path.join(CSRC, name)).read()):
        _device_sources(os.path.basename(inc), seen)
    return seen


def test_hashes_cover_the_kernels_sources():
    assert _device_sources("ctf_filter.cu", set()) <= set(bench.EXACT_SOURCES)
    assert _device_sources("ctf_mlp_ws2.cu", set()) <= set(bench.LEARNED_SOURCES)

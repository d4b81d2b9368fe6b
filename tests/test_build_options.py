"""Compile-time options of the kernels (MIRRES_NVCC_FLAGS) that a build must not be made unsafe with."""
import os
import subprocess

import pytest

from paper_2406_16360_gb300 import build as B


def _preprocessed(unit, *flags):
    r = subprocess.run([B.nvcc()] + B.ARCH + ["-std=c++17", "-I", B.CSRC, "-I", B.INCLUDE, *flags, "-E",
                                              os.path.join(B.CSRC, unit)], capture_output=True, text=True, check=True)
    return r.stdout


@pytest.mark.parametrize("flags", [(), ("-DMR_DFS_NODES=0",), ("-DMR_DFS_NODES=1",)])
def test_the_traversal_reads_the_64_byte_nodes(flags):
    """the builders' 48-byte records (no child codes) are never handed to a traversal"""
    lines = [ln.strip() for ln in _preprocessed("abi.cu", *flags).splitlines() if ln.strip().startswith("d.nodes =")]
    assert lines == ["d.nodes = s->dnodes;"]

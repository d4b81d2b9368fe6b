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


@pytest.mark.parametrize("flag,message", [("-DMR_PEND=1", "two leaves aside"), ("-DMR_PEND=0", "two leaves aside"),
                                          ("-DMR_REFILL_STEPS=0", "every second visit"),
                                          ("-DMR_REFILL_STEPS=7", "every second visit")])
def test_refilling_traversal_options_are_refused_out_of_range(tmp_path, flag, message):
    """with room for one leaf a lane writes behind its column or never goes on; without a visit
    between refills no ray ends"""
    src = tmp_path / "unit.cu"
    src.write_text('#include "device.cuh"\n')
    r = subprocess.run([B.nvcc()] + B.ARCH + ["-std=c++17", "-I", B.CSRC, "-I", B.INCLUDE, flag, "-ptx", "-o",
                                              str(tmp_path / "unit.ptx"), str(src)], capture_output=True, text=True)
    assert r.returncode != 0 and message in r.stderr

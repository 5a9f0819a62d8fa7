"""Registers of kernels whose rate depends on how many of their blocks fit an SM, as
the compiler reports them (no GPU needed)."""
import os
import re
import subprocess

import pytest

from paper_2605_01086_gb300.build import ARCH, CSRC, INCLUDE, _nvcc


def _ptxas(src, tmp_path):
    if _nvcc() is None:
        pytest.skip("nvcc not found")
    r = subprocess.run([_nvcc(), *ARCH, "-O3", "-std=c++17", "-Xptxas", "-v", "-I", INCLUDE, "-I", CSRC, "-c",
                        os.path.join(CSRC, src), "-o", str(tmp_path / "x.o")], capture_output=True, text=True, check=True)
    return re.findall(r"entry function '(\S+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads.*?Used (\d+) registers",
                      r.stderr + r.stdout, re.S)


def test_block_adjoint_leaves_room_for_1024_threads(tmp_path):
    """k_backward: 65,536 registers of an SM over 1024 threads, and no spills."""
    found = _ptxas("backward.cu", tmp_path)
    assert len(found) == 3
    for name, stores, loads, regs in found:
        assert int(regs) <= 64 and int(stores) == 0 and int(loads) == 0, (name, regs, stores, loads)

"""The rules that choose a kernel's variant (csrc/dispatch.h), compiled for the host: which side
a call of given sizes takes, at the measured crossings and beyond."""

import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_28699_gb300", "csrc")
SOURCE = r"""
#include "dispatch.h"
extern "C" {
int repair_wide(long cells, int threads) { return wc::repair_wide(cells, threads); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("dispatch")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{CSRC}", "-o", str(d / "t.so"), str(d / "t.cpp")],
                   check=True)
    return ctypes.CDLL(str(d / "t.so"))


@pytest.mark.parametrize("cells,threads,wide", [(28, 1024, 1), (152, 1024, 1), (153, 1024, 0), (280, 512, 1), (448, 512, 0),
                                                (1216, 128, 1), (2800, 128, 0), (8400, 64, 0), (229376, 64, 0)])
def test_repair_ctas_are_wide_while_the_chip_is_half_full(lib, cells, threads, wide):
    """One warp per small cell left a few cells with long chains: 28 of 128 pages took 7.5 us, 4.8 before."""
    assert lib.repair_wide(ctypes.c_long(cells), threads) == wide

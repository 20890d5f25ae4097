"""Index and scheduling arithmetic of the kernels (csrc/pt_rules.h), compiled by the host compiler and run at sizes that no
GPU test reaches."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include "pt_rules.h"
using namespace ptgb;
extern "C" {
int64_t grid_warp_(unsigned b, unsigned n, unsigned t) { return grid_warp(b, n, t); }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "librules.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2511_13508_gb300", "csrc"),
                    str(d / "shim.cpp"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.grid_warp_.restype = ctypes.c_int64
    return L


@pytest.mark.parametrize("chain", [0, 7, 8, (1 << 27) - 1, 1 << 27, (1 << 27) + 9, (1 << 28) - 1])
def test_a_warp_per_chain_reaches_every_chain(rules, chain):
    """Blocks of 8 warps: chain c is warp c of the grid, up to the 2^28 chains of a context."""
    for lane in (0, 31):
        assert rules.grid_warp_(chain // 8, 256, chain % 8 * 32 + lane) == chain

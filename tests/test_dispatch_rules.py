"""The rules that choose between kernels (csrc/dispatch.cuh), compiled for the host."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_21244_gb300", "csrc")
SMS = 152
CLAIMED, ONCE_8, ONCE_32 = 0, 8, 32

STUB = r"""
#include "dispatch.cuh"
extern "C" int cells(int match, int64_t n_cells, int64_t n, int64_t sms) {
  return dsmc::cells_kernel(match != 0, n_cells, n, sms);
}
extern "C" int groups(int table, int64_t n_cells, int64_t n, int64_t sms) {
  return dsmc::groups_suit(table != 0, n_cells, n, sms);
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("dispatch")
    src, lib = d / "rules.cc", d / "rules.so"
    src.write_text(STUB)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + CSRC, str(src), "-o", str(lib)], check=True)
    so = ctypes.CDLL(str(lib))
    for f in (so.cells, so.groups):
        f.argtypes = [ctypes.c_int] + [ctypes.c_int64] * 3
    return so


@pytest.mark.parametrize("match,n_cells,n,want", [
    (1, 8 * SMS, 0, ONCE_32), (1, 8 * SMS + 1, 0, ONCE_8), (0, 8 * SMS, 0, ONCE_32), (0, 320 * SMS, 0, ONCE_8),
    (0, 320 * SMS + 1, 0, CLAIMED),
    # a direct call does not know its particles: dense cells cost the groups more, so it changes over earlier
    (1, 96 * SMS, 0, ONCE_8), (1, 96 * SMS + 1, 0, CLAIMED), (1, 18375, 0, CLAIMED),
    # a step does
    (1, 128 * SMS, 2500 * SMS, ONCE_8), (1, 128 * SMS + 1, 2500 * SMS, CLAIMED), (1, 96 * SMS, 2500 * SMS + 1, CLAIMED),
    (0, 320 * SMS, 10000 * SMS, ONCE_8), (0, 96 * SMS, 10000 * SMS + 1, CLAIMED),
    # what the tuned shapes are for
    (1, 10, -1, CLAIMED), (0, 10, -1, CLAIMED),
    # few cells: most lanes per cell, however dense
    (1, 1000, 500000, ONCE_32), (0, 1000, 8000000, ONCE_32), (1, 8 * SMS, 2**31 - 1, ONCE_32),
])
def test_cell_kernel(rules, match, n_cells, n, want):
    assert rules.cells(match, n_cells, n, SMS) == want


@pytest.mark.parametrize("table,n_cells,n,want", [
    (0, 64 * SMS, 20 * 64 * SMS, 1), (0, 64 * SMS + 1, 20 * 64 * SMS, 0), (1, 288 * SMS, 20 * 288 * SMS, 1),
    (1, 288 * SMS + 1, 20 * 288 * SMS, 0), (0, 100, 0, 1),
    # few cells with many particles are many pairs for one warp each
    (0, 1, 512, 1), (0, 1, 513, 0), (1, 1, 1000000, 0), (1, 100, 51200, 1), (1, 100, 51201, 0),
    # a gas that fills the chip
    (0, 64 * SMS, 4000 * SMS, 1), (0, 64 * SMS, 4000 * SMS + 1, 0), (1, 288 * SMS, 16000 * SMS, 1),
    (1, 288 * SMS, 16000 * SMS + 1, 0),
])
def test_pair_update_by_groups(rules, table, n_cells, n, want):
    assert rules.groups(table, n_cells, n, SMS) == want

"""Shape of the gradient kernel of rows of 513 to 8,192 columns, compiled by the host compiler, at every length of a row."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_05203_b200", "csrc")
SHIM = """
#include "wide_ring.cuh"
using namespace ef21;
extern "C" void shape(int ld, int* out) {
    const WideShape s = GRAD_WIDE_SHAPES[grad_wide_shape(ld)];
    const int all[6] = {s.threads, s.columns, s.groups, s.rows, grad_wide_stages(s.groups, s.rows, ld), GRAD_WIDE_SMEM};
    for (int i = 0; i < 6; ++i) out[i] = all[i];
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    folder = tmp_path_factory.mktemp("ring")
    source, out = folder / "shim.cpp", folder / "shim.so"
    source.write_text(SHIM)
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", str(source), "-o", str(out)], check=True)
    return ctypes.CDLL(str(out))


def test_every_row_length_has_two_stages_in_flight(lib):
    out = (ctypes.c_int * 6)()
    for ld in range(516, 8193, 4):
        lib.shape(ld, out)
        threads, columns, groups, rows, stages, smem = out
        assert 4 * threads * columns >= ld and rows in (2, 4, 8), ld                # every column is some thread's
        assert 2 <= stages <= 8 and groups * stages * rows * ld * 4 <= smem, ld

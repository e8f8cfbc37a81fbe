"""Shape of the gradient kernel of rows of 513 to 8,192 columns, at every length of a row, and what its ring waits for when it stops early;
compiled by the host compiler."""
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
    const int all[8] = {s.threads, s.columns, s.groups, s.rows, grad_wide_stages(s.groups, s.rows, ld), GRAD_WIDE_SMEM, grad_wide_ring_bytes(s, ld),
                        grad_wide_smem_bytes(s, ld)};
    for (int i = 0; i < 8; ++i) out[i] = all[i];
}
// the stages and parities that are waited for, in `out`; returns how many
extern "C" int settle(int issued, int stages, int* out) {
    int n = 0;
    grad_wide_settle(issued, stages, [&](int stage, unsigned parity) { out[2 * n] = stage; out[2 * n + 1] = (int)parity; ++n; });
    return n;
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
    out = (ctypes.c_int * 8)()
    for ld in range(516, 8193, 4):
        lib.shape(ld, out)
        threads, columns, groups, rows, stages, smem, ring, total = out
        assert 4 * threads * columns >= ld and rows in (2, 4, 8), ld                # every column is some thread's
        assert 2 <= stages <= 8 and groups * stages * rows * ld * 4 == ring <= smem, ld
        assert total - ring >= (groups - 1) * ld * 4 and total <= smem + 8192, ld      # the groups' sums lie where no copy lands


def test_a_stop_waits_for_every_copy_under_way(lib):
    out = (ctypes.c_int * 16)()
    for stages in range(1, 9):
        for batches in range(0, 40):
            for stop in range(0, batches + 1):                # batches taken when the group stops; it fetches nothing more
                issued, phase = min(stages, batches), {}
                for taken in range(stop):
                    issued += issued < batches
                for b in range(issued):
                    phase[b % stages] = b // stages
                n = lib.settle(issued, stages, out)
                assert {out[2 * i]: out[2 * i + 1] for i in range(n)} == {s: u % 2 for s, u in phase.items()} and n == len(phase)

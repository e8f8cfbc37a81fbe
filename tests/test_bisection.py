"""The bisection that the selections of few entries start from, compiled by the host compiler: it ends, within 32 steps, on every set of keys
(all 32-bit patterns are entries a caller can pass, a NaN with all bits set among them) and its floor does what the selections rely on."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_05203_b200", "csrc")
SHIM = """
#include "bisect.cuh"
// floor and top over n keys as the kernels take them, with a limit of its own on the counts; returns the number of counts, -1 beyond it
extern "C" int search(const unsigned* keys, int n, int need, unsigned floor, unsigned top, unsigned* out) {
    int counts = 0;
    struct Endless {};
    try {
        *out = ef21::bisect_floor(floor, top, need, [&](unsigned key) {
            if (++counts > 1000) throw Endless();
            int c = 0;
            for (int i = 0; i < n; ++i) c += keys[i] >= key ? 1 : 0;
            return c;
        });
    } catch (Endless) { return -1; }
    return counts;
}
extern "C" int limit(int threads, int d, int alone, int grad) { return ef21::few_limit(threads, d, alone, grad); }
extern "C" unsigned middle(unsigned floor, unsigned top) { return ef21::bisect_middle(floor, top); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    folder = tmp_path_factory.mktemp("bisect")
    source, out = folder / "shim.cpp", folder / "shim.so"
    source.write_text(SHIM)
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-shared", "-fPIC", f"-I{CSRC}", str(source), "-o", str(out)], check=True)
    loaded = ctypes.CDLL(str(out))
    loaded.middle.restype = ctypes.c_uint
    loaded.middle.argtypes = [ctypes.c_uint, ctypes.c_uint]
    loaded.search.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_uint, ctypes.c_uint, ctypes.c_void_p]
    return loaded


EDGES = [0, 1, 2, 0x7fffffff, 0x80000000, 0x80000001, 0xff000000, 0xfffffffe, 0xffffffff]


def test_middle_lies_above_the_floor(lib):
    rng = np.random.default_rng(1)
    keys = EDGES + [int(v) for v in rng.integers(0, 1 << 32, 200)]
    for floor in keys:
        for top in keys:
            if floor < top:
                assert lib.middle(floor, top) == floor + (top - floor + 1) // 2


def _keys(kind, n, rng):
    keys = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
    if kind == "normal":                                  # magnitudes as the kernels hold them, rotated left by one
        keys = rng.standard_normal(n).astype(np.float32).view(np.uint32)
        keys = (keys << np.uint32(1)) | (keys >> np.uint32(31))
    elif kind == "idle":                                  # most threads without an entry
        keys[rng.permutation(n)[:n - n // 4]] = 0
    elif kind == "edges":
        keys = rng.choice(np.array(EDGES, np.uint32), n)
    elif kind == "one":
        keys[:] = 0
    elif kind == "equal":
        keys[:] = 0x7f800000
    return keys.astype(np.uint32)


@pytest.mark.parametrize("kind", ["any", "normal", "idle", "edges", "one", "equal"])
@pytest.mark.parametrize("top_key", [None, 0, 1, 0xfffffffe, 0xffffffff], ids=["as-drawn", "0", "1", "fffffffe", "ffffffff"])
def test_search_ends_and_its_floor_holds(lib, kind, top_key):
    rng = np.random.default_rng(2)
    for n in (32, 256, 512, 1024):
        for need in (1, 2, 7, n // 8, n // 4):
            keys = _keys(kind, n, rng)
            if top_key is not None:
                keys[rng.integers(n)] = top_key
            out = ctypes.c_uint()
            counts = lib.search(keys.ctypes.data, n, need, int(keys.min()), int(keys.max()), ctypes.byref(out))
            assert 0 <= counts <= 32, (n, need)
            reach = int((keys >= np.uint32(out.value)).sum())
            assert reach >= need, (n, need)
            if reach > need + need // 4 + 4:              # ties: nothing above has enough
                assert out.value == 0xffffffff or int((keys > np.uint32(out.value)).sum()) < need, (n, need)


@pytest.mark.parametrize("threads,first,last", [(256, 1, 2048), (512, 2049, 8192), (512, 513, 8192), (1024, 8193, 16384)])
def test_limit_of_few_entries(lib, threads, first, last):
    """Never more than a quarter of the threads (more of them need not have an entry to count), and not where a histogram was measured to be
    faster: many vectors, us with it and without, in bisect.cuh."""
    for d in range(first, last + 1):
        for grad in (0, 1):
            crowded, alone = lib.limit(threads, d, 0, grad), lib.limit(threads, d, 1, grad)
            assert 1 <= crowded <= alone <= threads // 4
    for slower in ((1024, 16384, 0, 0, 192), (1024, 9000, 0, 0, 128), (512, 8192, 0, 0, 112), (512, 2100, 0, 0, 64), (256, 2048, 0, 0, 64), (256, 300, 0, 0, 32),
                   (1024, 9000, 1, 0, 192), (512, 8192, 1, 0, 128), (512, 4000, 1, 0, 96), (256, 1000, 1, 0, 64), (512, 1500, 1, 1, 128)):
        assert lib.limit(*slower[:4]) < slower[4]

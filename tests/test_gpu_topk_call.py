"""topk() by its native call and by the general one: the same results and the same refusals."""
import ctypes
import importlib.util
import os
import shutil
import subprocess
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2106_05203_b200 import binding
    return binding


@pytest.mark.parametrize("batch,d,k", [(1, 1, 1), (1, 1000, 10), (3, 257, 257), (20, 70001, 700), (2, 800001, 8000), (65536 - 1, 3, 1), (2, 1048576, 600000)])
def test_same_results(B, batch, d, k):
    v = torch.randn(batch, d, device="cuda")
    native, general = B._topk_call(v, k), B.topk(v, k, torch.cuda.current_stream())
    assert type(native) is tuple
    for a, b in zip(native, general):
        assert a.dtype == b.dtype and a.shape == b.shape and a.stride() == b.stride() and torch.equal(a, b)
    if batch == 1:
        assert all(torch.equal(a, b) for a, b in zip(B.topk(v[0], k), native))
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):                       # the current stream is taken, whichever it is
        other = B.topk(v, k)
    stream.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(other, native))


def test_views_and_parameters(B):
    base = torch.randn(3, 5001, device="cuda")
    row = base[1]                                          # contiguous, not aligned
    order = torch.sort(row.abs(), descending=True, stable=True).indices[:50].sort().values
    assert torch.equal(B.topk(row, 50)[0][0].long(), order)
    p = torch.nn.Parameter(base)                           # (a subclass: the general call)
    idx, val = B.topk(p.requires_grad_(), 50)
    assert torch.equal(idx[1].long(), order) and not val.requires_grad


def test_refusals(B):
    v = torch.randn(4, 100, device="cuda")
    for bad in (v.t(), v.double(), v.cpu(), v[:, ::2]):
        with pytest.raises(TypeError):
            B.topk(bad, 3)
    for k in (0, -1, 101):
        with pytest.raises((B.Ef21Error, RuntimeError)):
            B.topk(v, k)
    with pytest.raises((ValueError, B.Ef21Error)):
        B.topk(v.view(2, 2, 100), 3)
    with pytest.raises(B.Ef21Error):
        B.topk(torch.empty(0, 10, device="cuda"), 3)
    batched = torch.func.vmap(lambda r: B.topk(r, 3)[1])
    with pytest.raises(RuntimeError):
        batched(v)


# an entry that comes back when another thread has set `seen`, with an error after two seconds
WAITING_ENTRY = """
#include <stddef.h>
#include <stdint.h>
#include <unistd.h>
extern "C" { volatile int entered = 0, seen = 0; }
extern "C" size_t bytes(int32_t, int64_t, int32_t) { return 64; }
extern "C" int entry(const float*, int32_t, int64_t, int32_t, int32_t*, float*, void*, size_t, void*) {
    entered = 1;
    for (int ms = 0; ms < 2000 && !seen; ++ms) usleep(1000);
    return seen ? 0 : 4;
}
"""


def test_other_threads_run_while_the_call_waits(B, tmp_path):
    (tmp_path / "entry.cpp").write_text(WAITING_ENTRY)
    subprocess.run([os.environ.get("CXX", "g++"), "-shared", "-fPIC", str(tmp_path / "entry.cpp"), "-o", str(tmp_path / "entry.so")], check=True)
    lib = ctypes.CDLL(str(tmp_path / "entry.so"))
    path = str(tmp_path / "_topk_call.so")                  # a copy, whose entry points are its own
    shutil.copy(os.path.join(os.path.dirname(B.__file__), "_topk_call.so"), path)
    spec = importlib.util.spec_from_file_location("_topk_call", path)
    module = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(module)
    module.set_entry(*(ctypes.cast(f, ctypes.c_void_p).value for f in (lib.bytes, lib.entry)))
    entered, seen = ctypes.c_int.in_dll(lib, "entered"), ctypes.c_int.in_dll(lib, "seen")

    def other():
        while not entered.value:
            pass
        seen.value = 1

    thread = threading.Thread(target=other)
    thread.start()
    out = module.topk(torch.randn(2, 100, device="cuda"), 3)
    thread.join()
    assert type(out) is tuple

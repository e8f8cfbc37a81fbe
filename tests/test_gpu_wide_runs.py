"""Runs on rows of 513 to 8,192 columns (gradient tiles through a ring that later iterations of a call fill ahead of time, gradients
formed by the selecting cluster), and the selection of few entries in one block: at the edges of their shapes."""
import numpy as np
import pytest
import torch

import ef21_inputs as inputs
from gpu_util import dev, lockstep, make_gpu, make_oracle_state

pytestmark = pytest.mark.gpu

# d, n, rows, k: clusters of 8, 4, 2 and 1 forming blocks; k up to and beyond a quarter of 512 threads; tiles from one row on; up to 40
# tiles per worker and more
SHAPES = [(513, 3, 40, 5), (700, 2, 900, 7), (1025, 37, 500, 20), (2047, 75, 300, 128), (2048, 75, 160, 129), (2049, 9, 70, 1), (4100, 4, 700, 41),
          (5001, 20, 900, 50), (5121, 20, 900, 51), (6144, 9, 1500, 61), (6145, 40, 300, 60), (8192, 5, 333, 128)]


def _workload(d, n, rows, k):
    return inputs.make_logistic("wide", n=n, d=d, N=rows, k=k, seed=d + n, features="bernoulli", density=0.1, gamma=0.05, T=10)


@pytest.mark.parametrize("d,n,rows,k", SHAPES)
def test_wide_runs_track_the_oracle(d, n, rows, k, oracle32):
    from paper_2106_05203_b200 import binding as B
    w = _workload(d, n, rows, k)
    h = make_gpu(w)
    st = make_oracle_state(oracle32, w)
    h.init(B.INIT_COMPRESSED)
    st.init(0)
    lockstep(h, st, oracle32, w, 4)
    assert h.last_path == B.PATH_LAUNCHES and h.poll() == 0


@pytest.mark.parametrize("variant", [0, 1, 2])
@pytest.mark.parametrize("d,n,rows,k", SHAPES[:4] + SHAPES[7:])
def test_one_call_gives_the_bits_of_many(d, n, rows, k, variant):
    from paper_2106_05203_b200 import binding as B
    w = _workload(d, n, rows, k)
    states = []
    for calls, steps in ((1, 7), (7, 1)):
        h = make_gpu(w)
        h.set_variant(variant)
        h.init(B.INIT_ZERO)
        for _ in range(calls):
            h.step(steps)
        assert h.poll() == 0
        states.append(h.get_state())
    for a, b in zip(*states):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))


@pytest.mark.parametrize("d,n,rows,k", [SHAPES[1], SHAPES[4], (2049, 9, 7000, 1), (5001, 20, 9000, 50), (5121, 20, 9000, 51), (6145, 40, 3000, 60)])
def test_a_gradient_kernel_that_gives_up_leaves_nothing_behind(d, n, rows, k, oracle32):
    # its first copies of rows are under way when it stops; the kernels behind it get its shared memory
    from paper_2106_05203_b200 import binding as B
    w = _workload(d, n, rows, k)
    h = make_gpu(w)
    st = make_oracle_state(oracle32, w)
    h.init(B.INIT_COMPRESSED)
    st.init(0)
    saved = h.get_state()[:3]
    for _ in range(3):
        h.selftest_bounded_wait(1)
        h.step(1)
    assert h.poll() == 5
    h.set_state(*saved)
    h.clear_status()
    lockstep(h, st, oracle32, w, 2)
    assert h.poll() == 0


# blocks of 256, 512 and 1,024 threads: k at a quarter of them and one more, lengths at the values a thread holds
@pytest.mark.parametrize("kind", ["gauss", "ties", "signs", "few nonzero", "zeros", "spread"])
@pytest.mark.parametrize("batch,d,k", [(3, 7, 7), (3, 257, 64), (5, 2048, 64), (5, 2048, 65), (3, 2049, 128), (3, 8192, 128), (3, 8192, 129), (150, 8193, 256),
                                       (150, 16384, 256), (150, 16384, 257), (150, 16385, 20), (2, 5000, 1), (3, 8192, 118), (3, 8192, 119),
                                       (150, 16384, 155), (150, 16384, 156), (3, 300, 32), (3, 300, 33)])
def test_few_entries_of_short_vectors(batch, d, k, kind, oracle32):
    from paper_2106_05203_b200 import binding as B
    rng = np.random.default_rng(d + k)
    v = rng.standard_normal((batch, d), dtype=np.float32)
    if kind == "ties":
        v = np.round(v * 2).astype(np.float32) * np.float32(0.5)
    elif kind == "signs":
        v = np.sign(v).astype(np.float32)
    elif kind == "few nonzero":
        v *= rng.random((batch, d)) < 0.5 * k / d
    elif kind == "zeros":
        v *= np.float32(0)                                     # of both signs
    elif kind == "spread":
        v = (v * np.exp2(rng.integers(-140, 100, (batch, d)).astype(np.float64))).astype(np.float32)      # subnormals among them
    idx, val = B.topk(dev(v), k)
    for i in sorted({0, batch // 2, batch - 1}):
        oi, ov = oracle32.topk(v[i], k)
        np.testing.assert_array_equal(idx[i].cpu().numpy(), oi)
        np.testing.assert_array_equal(val[i].cpu().numpy().view(np.uint32), ov.view(np.uint32))


# clusters of 2, 4, 8 and 16 blocks; k up to what the cluster's floors are used for and one more; the large entries in one block's
# share (more candidates than it lists), ties at the cut in several blocks
@pytest.mark.parametrize("kind", ["gauss", "ties", "signs", "layers", "bf16", "few nonzero"])
@pytest.mark.parametrize("batch,d,k", [(1, 16384, 1), (40, 16385, 408), (3, 65537, 700), (20, 70001, 816), (20, 70001, 817), (2, 94209, 1024), (2, 376833, 1024),
                                       (70, 30000, 39), (70, 30000, 40), (37, 60000, 79), (37, 60000, 80),
                                       (1, 376833, 1025), (1, 753664, 753)])
def test_few_entries_in_a_cluster(batch, d, k, kind, oracle32):
    from paper_2106_05203_b200 import binding as B
    rng = np.random.default_rng(d + k)
    v = rng.standard_normal((batch, d), dtype=np.float32)
    if kind == "ties":
        v = np.round(v * 4).astype(np.float32) * np.float32(0.25)
    elif kind == "signs":
        v = np.sign(v).astype(np.float32)
    elif kind == "layers":
        v[:, d // 3:d // 3 + max(2 * k, 1500)] *= np.float32(100)
    elif kind == "bf16":
        v = (v.view(np.uint32) & np.uint32(0xffff0000)).view(np.float32)
    elif kind == "few nonzero":
        v *= rng.random((batch, d)) < 0.5 * k / d
    idx, val = B.topk(dev(v), k)
    for i in sorted({0, batch // 2, batch - 1}):
        oi, ov = oracle32.topk(v[i], k)
        np.testing.assert_array_equal(idx[i].cpu().numpy(), oi)
        np.testing.assert_array_equal(val[i].cpu().numpy().view(np.uint32), ov.view(np.uint32))


@pytest.mark.parametrize("variant", [0, 1, 2])
@pytest.mark.parametrize("n,d,k", [(20, 70001, 700), (8, 95620, 95), (3, 376833, 1000)])
def test_rounds_with_few_entries_in_a_cluster(n, d, k, variant):
    from paper_2106_05203_b200 import binding as B
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d)
    states = []
    V = [torch.randn(n, d, device="cuda", generator=gen) * (1 + 3 * t) for t in range(3)]
    V[1][0, d // 2:d // 2 + 2000] *= 50
    for algorithm in (0, 1):
        h = B.EF21(n, d, k, 0.05)
        h.set_variant(variant)
        h.set_topk_algorithm(algorithm)
        h.init_grads(None, B.INIT_ZERO)
        for v in V:
            h.step_grads(v, 2)
        assert h.poll() == 0
        states.append(h.get_state())
    for a, b in zip(*states):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))

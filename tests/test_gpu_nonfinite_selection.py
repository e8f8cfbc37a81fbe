"""Selections from vectors with infinities and NaN of both signs and of any payload, all bits set among them (memory filled with 0xff, an
integer -1 seen as a float): a selection compares bit patterns, so the oracle has one answer for each, bit for bit.  Every path of the
standalone Top-k, the initial g_i, and EF21+."""
import numpy as np
import pytest
import torch

from gpu_util import dev

pytestmark = pytest.mark.gpu

SPECIAL = np.array([0xffffffff, 0x7fffffff, 0xffc00000, 0x7fc00000, 0x7f800001, 0xff800001, 0x7f800000, 0xff800000], np.uint32)
KINDS = ["one", "all bits set", "mixed", "many", "sparse", "filled"]


def _vectors(kind, batch, d, k, seed):
    rng = np.random.default_rng(seed)
    v = rng.standard_normal((batch, d), dtype=np.float32)
    bits = v.view(np.uint32)
    for i in range(batch):
        if kind == "one":                                    # the only entry beyond the finite ones, the key with all bits set
            bits[i, rng.integers(d)] = 0xffffffff
        elif kind == "all bits set":
            bits[i, rng.permutation(d)[:max(1, k // 2)]] = 0xffffffff
        elif kind == "mixed":
            at = rng.permutation(d)[:max(1, k // 2)]
            bits[i, at] = rng.choice(SPECIAL, at.size)
        elif kind == "many":                                 # more than the message holds
            at = rng.permutation(d)[:min(d, 2 * k)]
            bits[i, at] = rng.choice(SPECIAL, at.size)
        elif kind == "sparse":                               # nine tenths zeros: most threads have no other entry
            bits[i, rng.random(d) < 0.9] = 0
            bits[i, rng.integers(d)] = 0xffffffff
        else:
            bits[i] = 0xffffffff
    return v


# one block of 256, 512 and 1,024 threads with few entries and with more; clusters of 2, 4, 8 and 16 blocks, by way of floors and without;
# the streaming pass
SHAPES = [(3, 5, 1), (3, 200, 2), (3, 255, 60), (2, 1000, 10), (3, 2048, 65), (3, 2049, 128), (150, 16384, 256), (1, 16384, 1), (3, 65537, 700),
          (20, 70001, 700), (1, 81822, 818), (2, 376833, 1024), (1, 753664, 753), (1, 753665, 753), (20, 262145, 262)]


def _check(idx, val, v, k, oracle):
    for i in sorted({0, v.shape[0] // 2, v.shape[0] - 1}):
        oi, ov = oracle.topk(v[i], k)
        np.testing.assert_array_equal(idx[i].cpu().numpy(), oi)
        np.testing.assert_array_equal(val[i].view(torch.int32).cpu().numpy().view(np.uint32), ov.view(np.uint32))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("batch,d,k", SHAPES)
def test_topk(batch, d, k, kind, oracle32):
    from paper_2106_05203_b200 import binding as B
    v = _vectors(kind, batch, d, k, d + k)
    V = dev(v)
    _check(*B.topk(V, k), v, k, oracle32)
    if batch <= 64 and batch * -(-d // 4096) <= 16384:
        idx, val = torch.empty(batch, k, dtype=torch.int32, device="cuda"), torch.empty(batch, k, device="cuda")
        B.topk_static(V, k, idx, val)
        _check(idx, val, v, k, oracle32)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n,d,k", [(3, 200, 2), (20, 70001, 700), (3, 300000, 300)])
def test_initial_messages(n, d, k, kind, oracle32):
    from paper_2106_05203_b200 import binding as B
    v = _vectors(kind, n, d, k, d)
    h = B.EF21(n, d, k, 0.05)
    h.init_grads(dev(v), B.INIT_COMPRESSED)
    v.view(np.uint32)[np.isnan(v)] = 0x7fffffff              # the difference with g_i = 0 is selected from: the device's own NaN
    _, _, gi, idx, val = h.get_state()
    _check(idx, val, v, k, oracle32)
    kept = torch.zeros_like(gi, dtype=torch.bool).scatter_(1, idx.long(), True)
    assert not gi[~kept].any()
    assert h.poll() == 6


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n,d,k", [(3, 200, 2), (20, 70001, 700), (20, 262147, 2621), (19, 263168, 263)])
def test_plus(n, d, k, kind):
    """EF21+, whose plain selection takes the gradients unchanged: one step behind two finite ones, against the multi-pass selection."""
    from paper_2106_05203_b200 import binding as B
    good = [dev(np.random.default_rng(t).standard_normal((n, d), dtype=np.float32)) for t in range(2)]
    bad = dev(_vectors(kind, n, d, k, d))
    states = []
    for algorithm in (0, 1):
        h = B.EF21(n, d, k, 0.05)
        h.set_variant(B.VARIANT_EF21_PLUS)
        h.set_topk_algorithm(algorithm)
        h.init_grads(None, B.INIT_ZERO)
        for V in good:
            h.step_grads(V, 1)
        assert h.poll() == 0
        h.step_grads(bad, 1)
        states.append((h.get_plus_choice(), h.get_state()))
        assert h.poll() == 6
    np.testing.assert_array_equal(states[0][0], states[1][0])
    for a, b in zip(states[0][1], states[1][1]):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))

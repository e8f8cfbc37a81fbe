"""Standalone Top-k at the edges of its dispatch (one cluster per vector, streaming pass, second read of the regions),
against the oracle, bit for bit."""
import numpy as np
import pytest

from gpu_util import dev

pytestmark = pytest.mark.gpu

# batch, d, k, kind.  47,104 floats fill a block's share of a cluster; 262,144 is the shortest vector of the streaming pass,
# which takes what no cluster of 16 blocks holds and large batches.
CASES = [
    (2, 2048, 20, "gauss"), (2, 2049, 2049, "gauss"), (3, 8192, 1, "gauss"), (3, 8193, 81, "ties"), (1, 16384, 5000, "gauss"),
    (2, 47104, 470, "bf16"), (2, 47105, 47104, "gauss"), (20, 94209, 94, "gauss"), (1, 376833, 3768, "ties"), (1, 753664, 75366, "gauss"),
    (1, 753665, 753, "gauss"), (3, 800001, 8000, "bf16"), (2, 900001, 90000, "gauss"), (1, 1048576, 524288, "gauss"),
    (20, 300000, 3000, "gauss"), (20, 262145, 262, "layers"), (65, 1048576, 1048, "gauss"), (1, 1000003, 900000, "ties"),
]


@pytest.mark.parametrize("batch,d,k,kind", CASES, ids=[f"{b}x{d}-k{k}-{kind}" for b, d, k, kind in CASES])
def test_topk_dispatch_edges(batch, d, k, kind, oracle32):
    from paper_2106_05203_b200 import binding as B
    rng = np.random.default_rng(d + k)
    v = rng.standard_normal((batch, d), dtype=np.float32)
    if kind == "ties":
        v = np.round(v * 2).astype(np.float32) * np.float32(0.5)
    elif kind == "bf16":
        v = (v.view(np.uint32) & np.uint32(0xffff0000)).view(np.float32)
    elif kind == "layers":                                   # the large entries sit together: lists of single regions overflow
        v[:, d // 3:d // 3 + d // 50] *= np.float32(100)
    idx, val = B.topk(dev(v), k)
    for i in sorted({0, batch // 2, batch - 1}):
        oi, ov = oracle32.topk(v[i], k)
        np.testing.assert_array_equal(idx[i].cpu().numpy(), oi)
        np.testing.assert_array_equal(val[i].cpu().numpy().view(np.uint32), ov.view(np.uint32))


@pytest.mark.parametrize("variant,n,d,k", [(0, 3, 70001, 700), (2, 3, 70001, 700), (1, 3, 70001, 700), (0, 24, 300001, 3000),
                                           (2, 24, 300000, 300), (1, 24, 300001, 3000), (2, 24, 300001, 40000), (1, 3, 800001, 100000),
                                           (0, 17, 4194304, 4194)])
def test_rounds_on_the_long_paths(variant, n, d, k, oracle32):
    """State after rounds on supplied gradients (messages, state update, tile offsets of the aggregation), bit for bit."""
    import oracle as oracle_mod
    from paper_2106_05203_b200 import binding as B
    rng = np.random.default_rng(n + d)
    V = rng.standard_normal((n, d), dtype=np.float32)
    steps = 1 if n * d > 20_000_000 else 3
    h = B.EF21(n, d, k, 0.05)
    h.set_variant(variant)
    h.init_grads(None, B.INIT_ZERO)
    h.step_grads(dev(V), steps)
    if variant == B.VARIANT_EF:
        st = oracle_mod.EFState(oracle32, n, d, k, 0.05)
        st.init_from_grads(V)
        st.step_grads(V, steps)
        want = st.e
    else:
        st = oracle_mod.State(oracle32, n, d, k, 0.05)
        st.init(1)
        (st.plus_step_grads if variant == B.VARIANT_EF21_PLUS else st.step_grads)(V, steps)
        want = st.gi
    x, g, gi, _, _ = h.get_state_host()
    np.testing.assert_array_equal(gi.view(np.uint32), want.view(np.uint32))
    np.testing.assert_array_equal(x.view(np.uint32), st.x.view(np.uint32))
    if variant != B.VARIANT_EF:
        np.testing.assert_array_equal(g.view(np.uint32), st.g.view(np.uint32))
    assert h.poll() == 0


@pytest.mark.parametrize("n,d,k", [(16, 4194304, 40000), (24, 3000000, 12000), (64, 1200000, 12000)])
def test_larger_messages_stay_on_the_streaming_path(n, d, k):
    """Large batches of aligned vectors with up to 1 % of the entries per message: exact, and no vector needs a second look."""
    import torch
    from paper_2106_05203_b200 import binding as B
    gen = torch.Generator(device="cuda")
    gen.manual_seed(k)
    V = torch.randn(n, d, device="cuda", generator=gen)
    h = B.EF21(n, d, k, 0.05)
    h.init_grads(None, B.INIT_ZERO)
    h.step_grads(V, 1)
    assert h.fallback_count() == 0 and h.poll() == 0
    idx, val = h.get_state(messages=True)[3:5]
    for i in (0, n // 2, n - 1):
        order = torch.sort(V[i].abs(), descending=True, stable=True).indices[:k].sort().values
        assert torch.equal(idx[i].long(), order) and torch.equal(val[i], V[i][order])

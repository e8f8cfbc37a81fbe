"""EF21+ on long vectors: both selections and the distortions' sums from one pass.  Both branches, state zero, candidates that coincide (a tie
goes to the Markov compressor) and distortions that nearly do, terms beyond the range of 32 bits, crowded regions and masses of ties (the exact
fallback) -- against the oracle, or against the multi-pass selection with its ordered sums, bit for bit."""
import numpy as np
import pytest
import torch

import oracle as oracle_mod
from gpu_util import dev

pytestmark = pytest.mark.gpu


def _gradients(kind, n, d, k, steps, seed):
    rng = np.random.default_rng(seed)
    base = rng.standard_normal((n, d)).astype(np.float32)
    out = []
    for t in range(steps):
        if kind == "jumps":                       # some rounds keep the Markov compressor, others restart
            v = base * np.float32(1.0 if t % 3 else 25.0) + np.float32(0.01) * rng.standard_normal((n, d)).astype(np.float32)
        elif kind == "coincide":                  # k entries rule and change little, exactly: both compressors then send the same vector
            v = base * np.float32(1e-4)
            v[:, ::d // k][:, :k] = np.float32(8.0 + t / 8)
        elif kind == "near":                      # the two distortions differ in a late bit
            v = base.copy()
            v[:, 0] = np.float32(1e3 * (1 + t * 1e-3))
            v[:, 1] = np.float32(1e-3 * t)
        elif kind == "huge":                      # squares beyond 32 bits, and below
            v = base * np.float32(1e25 if t % 2 else 1e-25)
        elif kind == "crowded":                   # the large entries sit together
            v = base.copy()
            v[:, d // 3:d // 3 + 3000] *= np.float32(100 + t)
        else:                                     # ties
            v = np.sign(base) * np.float32(1 + t)
        out.append(v.astype(np.float32))
    return out


@pytest.mark.parametrize("kind", ["jumps", "coincide", "near", "huge", "crowded", "ties"])
@pytest.mark.parametrize("n,d,k", [(20, 262147, 2621), (19, 263168, 263), (24, 270004, 18000)])
def test_against_the_multi_pass_selection(n, d, k, kind):
    from paper_2106_05203_b200 import binding as B
    handles = []
    for algorithm in (0, 1):
        h = B.EF21(n, d, k, 0.05)
        h.set_variant(B.VARIANT_EF21_PLUS)
        h.set_topk_algorithm(algorithm)
        h.init_grads(None, B.INIT_ZERO)
        handles.append(h)
    seen = set()
    for t, v in enumerate(_gradients(kind, n, d, k, 5, d + k)):
        V = dev(v)
        for h in handles:
            h.step_grads(V, 2 if t == 3 else 1)
        np.testing.assert_array_equal(handles[0].get_plus_choice(), handles[1].get_plus_choice(), err_msg=f"step {t}")
        for a, b in zip(handles[0].get_state(), handles[1].get_state()):
            assert torch.equal(a.view(torch.int32), b.view(torch.int32)), t
        seen |= set(handles[0].get_plus_choice().tolist())
        if t == 0:
            assert seen == {0}                                      # g_i = 0: the candidates coincide
    assert handles[0].poll() == 0
    if kind == "jumps":
        assert seen == {0, 1}
    if kind == "ties":
        assert handles[0].fallback_count() > 0


def test_against_the_oracle(oracle32):
    from paper_2106_05203_b200 import binding as B
    n, d, k = 20, 262147, 2621
    h = B.EF21(n, d, k, 0.05)
    h.set_variant(B.VARIANT_EF21_PLUS)
    st = oracle_mod.State(oracle32, n, d, k, 0.05)
    h.init_grads(None, B.INIT_ZERO)
    st.init(1)
    for kind in ("jumps", "coincide"):
        for v in _gradients(kind, n, d, k, 4, 7):
            h.step_grads(dev(v), 1)
            st.plus_step_grads(v, 1)
            x, g, gi, li, lv = h.get_state_host()
            np.testing.assert_array_equal(h.get_plus_choice(), st.choice)
            np.testing.assert_array_equal(li, st.idx)
            for a, b in ((lv, st.val), (gi, st.gi), (g, st.g), (x, st.x)):
                np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))

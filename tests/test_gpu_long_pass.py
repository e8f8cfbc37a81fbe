"""The streaming pass over large batches of aligned rows (n d >= 2^26): the last region of a vector from four entries to all but
four of its 4,096, full regions only, candidates in the last entries, and a region with more candidates than its list holds --
against the oracle and, for all workers, against the multi-pass selection, bit for bit."""
import numpy as np
import pytest
import torch

import ef21_inputs as inputs
import oracle as oracle_mod

pytestmark = pytest.mark.gpu


def _vectors(n, d, crowded):
    base = torch.from_numpy(inputs.stress_vector(11, 0, d)).cuda()
    V = torch.stack([torch.roll(base, 4099 * i) * (1.0 + 0.01 * i) for i in range(n)])
    V[:, -3:] = torch.tensor([50.0, -60.0, 70.0], device="cuda")
    V[:, 0] = 80.0
    if crowded:
        V[1, 5 * 4096:6 * 4096] += 1000.0 * torch.sign(V[1, 5 * 4096:6 * 4096])
    return V.contiguous()


@pytest.mark.parametrize("variant", [0, 2])
@pytest.mark.parametrize("n,d,crowded", [(64, 1048580, False), (16, 4198396, True), (17, 4194432, False), (33, 2099200, False), (65, 1048576, True)])
def test_rounds_and_topk(n, d, crowded, variant, oracle32):
    from paper_2106_05203_b200 import binding as B
    k = d // 1000
    V = _vectors(n, d, crowded)
    handles = []
    for algorithm in (0, 1):
        h = B.EF21(n, d, k, 0.01)
        h.set_variant(variant)
        h.set_topk_algorithm(algorithm)
        h.init_grads(None, B.INIT_ZERO)
        h.step_grads(V, 2)
        h.step_grads(V, 1)
        assert h.poll() == 0
        handles.append(h)
    assert (handles[0].fallback_count() > 0) == crowded
    for a, b in zip(handles[0].get_state(), handles[1].get_state()):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    if variant == 0:
        _, _, gi, li, lv = handles[0].get_state()
        for i in (1, n - 1):
            solo = oracle_mod.State(oracle32, 1, d, k, 0.01)
            solo.init(1)
            solo.step_grads(V[i].cpu().numpy()[None, :], 3)
            np.testing.assert_array_equal(li[i].cpu().numpy(), solo.idx[0])
            np.testing.assert_array_equal(lv[i].cpu().numpy().view(np.uint32), solo.val[0].view(np.uint32))
            np.testing.assert_array_equal(gi[i].cpu().numpy().view(np.uint32), solo.gi[0].view(np.uint32))
        idx, val = B.topk(V, k)
        for i in (1, n - 1):
            oi, ov = oracle32.topk(V[i].cpu().numpy(), k)
            np.testing.assert_array_equal(idx[i].cpu().numpy(), oi)
            np.testing.assert_array_equal(val[i].cpu().numpy().view(np.uint32), ov.view(np.uint32))

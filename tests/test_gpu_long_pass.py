"""The streaming pass over large batches of aligned rows (n d >= 2^26): the last region of a vector from four entries to all but
four of its 4,096, full regions only, candidates in the last entries, and a region with more candidates than its list holds; then
groups of equal keys at the cut, in large batches and small --
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


# the k-th key belongs to a group of some hundreds to some thousands of entries (more than are ranked one against the other)
@pytest.mark.parametrize("n,d,step,k", [(64, 1048576, 2.0, 1048), (64, 1048576, 1.0, 8000), (3, 1048577, 2.0, 1500), (1, 4194304, 1.0, 4194), (5, 1048580, 0.125, 60000)])
def test_groups_of_equal_keys(n, d, step, k, oracle32):
    from paper_2106_05203_b200 import binding as B
    base = torch.from_numpy(inputs.stress_vector(12, 0, d)).cuda()
    V = torch.stack([torch.round(torch.roll(base, 4099 * i) / step) * step for i in range(n)]).contiguous()
    handles = []
    for algorithm in (0, 1):
        h = B.EF21(n, d, k, 0.01)
        h.set_topk_algorithm(algorithm)
        h.init_grads(None, B.INIT_ZERO)
        h.step_grads(V, 1)
        assert h.poll() == 0
        handles.append(h)
    assert handles[0].fallback_count() == 0
    for a, b in zip(handles[0].get_state(), handles[1].get_state()):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    _, _, _, li, lv = handles[0].get_state()
    oi, ov = oracle32.topk(V[n - 1].cpu().numpy(), k)
    np.testing.assert_array_equal(li[n - 1].cpu().numpy(), oi)
    np.testing.assert_array_equal(lv[n - 1].cpu().numpy().view(np.uint32), ov.view(np.uint32))
    group = int((V[n - 1].abs() == float(np.abs(ov).min())).sum())
    assert 256 < group < 8192

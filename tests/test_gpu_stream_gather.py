"""The streaming pass of long vectors that are not listed in one go: candidates of a region from none to all of its 1,024 entries (a
warp's buffer holds 160 and is emptied from 32 on), rows aligned and not, regions with a ragged end, ties at the cut on both sides of a
region's border, with and without lists -- messages and state bit for bit against the multi-pass selection, Top-k against a sort."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _vectors(n, d, crowd):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d + crowd)
    V = torch.randn(n, d, device="cuda", generator=gen)
    V[0] = torch.round(V[0] * 4) / 4                              # groups of equal keys at the cut
    for r, per in enumerate((0, 31, 32, 33, 127, 128, 129, 159, 160, 161, 192, crowd)):
        lo = (3 + 5 * r) * 1024
        V[1, lo:lo + 1024] *= 0.001
        V[1, lo + 1024 - per:lo + 1024] = 40.0 + torch.rand(per, device="cuda", generator=gen)
    V[:, -1] = 70.0
    return V.contiguous()


@pytest.mark.parametrize("variant", [0, 2])
@pytest.mark.parametrize("n,d,k,crowd", [(20, 262144, 2621, 256), (20, 262147, 2621, 257), (19, 263169, 30000, 1024), (20, 263168, 50000, 1023),
                                         (20, 300001, 150000, 512), (20, 300004, 300, 1024),
                                         # the shortest vectors of the pass, with smaller samples (clusters of them would run in turn)
                                         (38, 131072, 131, 129), (40, 135001, 1350, 1024), (75, 131073, 20000, 300), (19, 262143, 60000, 512)])
def test_rounds_and_topk(n, d, k, crowd, variant):
    from paper_2106_05203_b200 import binding as B
    V = _vectors(n, d, crowd)
    handles = []
    for algorithm in (0, 1):
        h = B.EF21(n, d, k, 0.05)
        h.set_variant(variant)
        h.set_topk_algorithm(algorithm)
        h.init_grads(None, B.INIT_ZERO)
        h.step_grads(V, 2)
        assert h.poll() == 0
        handles.append(h)
    for a, b in zip(handles[0].get_state(), handles[1].get_state()):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    idx, val = B.topk(V, k)
    for i in (0, 1, n - 1):
        order = torch.sort(V[i].abs(), descending=True, stable=True).indices[:k].sort().values
        assert torch.equal(idx[i].long(), order) and torch.equal(val[i], V[i][order])


# vectors that are redone: clusters of eight with the vector in shared memory up to 376,832 entries, above it from global memory
@pytest.mark.parametrize("kind", ["zeros", "few nonzero", "signs", "one vector"])
@pytest.mark.parametrize("variant", [0, 2])
@pytest.mark.parametrize("n,d,k", [(38, 131072, 1310), (38, 131073, 20000), (19, 262143, 262), (19, 376832, 3768), (19, 376833, 3768)])
def test_redone_vectors(n, d, k, variant, kind):
    from paper_2106_05203_b200 import binding as B
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d)
    V = torch.randn(2, n, d, device="cuda", generator=gen)
    if kind == "zeros":
        V[1].zero_()
    elif kind == "few nonzero":
        V *= torch.rand(2, n, d, device="cuda", generator=gen) < 0.5 * k / d
    elif kind == "signs":
        V = V.sign()
    else:
        V[:, n // 2] = 1.0
    states = []
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

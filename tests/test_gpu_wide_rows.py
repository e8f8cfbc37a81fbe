"""Local gradients of rows wider than 512 columns: register shares, row batches and tiles at their edges, against fp64."""
import numpy as np
import pytest
import torch

from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,rows", [(513, 3, 40), (1024, 2, 17), (1025, 5, 333), (2048, 20, 801), (2049, 3, 9), (4095, 7, 1500),
                                      (5001, 20, 6000), (5121, 4, 5), (6145, 2, 301), (8192, 10, 2000), (8193, 3, 100)])
@pytest.mark.parametrize("objective", [0, 1])
def test_wide_rows(d, n, rows, objective):
    from paper_2106_05203_b200 import binding as B
    rng = np.random.default_rng(d)
    A, x = rng.standard_normal((rows, d), dtype=np.float32), (rng.standard_normal(d) / np.sqrt(d)).astype(np.float32)
    y = np.where(rng.random(rows) < 0.5, -1, 1).astype(np.float32)
    off = np.sort(np.r_[0, rng.integers(0, rows + 1, n - 1), rows])            # ragged, some shards may be empty
    h = B.EF21(n, d, 1, 0.1, 0.05, total_rows=rows)
    h.set_objective(objective)
    h.load_shards(dev(A), dev(y), off)
    h.set_x(dev(x))
    got = h.local_grads().cpu().numpy().astype(np.float64)
    x64 = x.astype(np.float64)
    z = A.astype(np.float64) @ x64
    rho = 2 * (z - y) if objective else -y / (1 + np.exp(y * z))
    for i in range(n):
        a, b = off[i], off[i + 1]
        want = (rho[a:b] @ A[a:b].astype(np.float64)) / max(1, b - a) + 2 * np.float64(np.float32(0.05)) * x64 / (1 + x64 ** 2) ** 2
        assert np.linalg.norm(got[i] - want) <= 1e-5 * np.linalg.norm(want), i
    f = h.eval()[0]
    loss = (z - y) ** 2 if objective else np.log1p(np.exp(-y * z))
    f_want = np.mean([loss[off[i]:off[i + 1]].mean() if off[i + 1] > off[i] else 0.0 for i in range(n)])
    f_want += np.float64(np.float32(0.05)) * np.sum(x64 ** 2 / (1 + x64 ** 2))
    assert abs(f - f_want) <= 1e-5 * abs(f_want)
    assert h.poll() == 0


@pytest.mark.parametrize("d,tau", [(700, 3), (3000, 64), (6000, 200)])
def test_wide_sampled_rows_in_order_are_the_full_shard(d, tau):
    from paper_2106_05203_b200 import binding as B
    rng = np.random.default_rng(d + tau)
    n = 6
    A = dev(rng.standard_normal((n * tau, d), dtype=np.float32))
    y = dev(np.where(rng.random(n * tau) < 0.5, -1, 1).astype(np.float32))
    states = []
    for sampled in (False, True):
        h = B.EF21(n, d, 4, 0.05, 0.1, total_rows=n * tau)
        h.load_shards(A, y, [i * tau for i in range(n + 1)])
        h.init(B.INIT_ZERO)
        if sampled:
            h.step_minibatch(torch.arange(tau, dtype=torch.int32, device="cuda").repeat(n, 1).contiguous())
        else:
            h.step(1)
        states.append(h.get_state_host())
        assert h.poll() == 0
    for a, b in zip(*states):
        np.testing.assert_allclose(a, b, rtol=1e-5, atol=1e-7)

"""Aggregation of vectors beyond the table's range where workers name the same coordinates: none, some, all of them; few workers with many
entries in a tile (resolved worker by worker) and many with few (resolved by looking through the list) -- bit for bit against the oracle."""
import numpy as np
import pytest

import oracle as oracle_mod
from gpu_util import assert_state_bitwise, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shared", [0.0, 0.3, 1.0])
@pytest.mark.parametrize("n,d,k", [(2, 20001, 1500), (5, 40000, 1000), (20, 20001, 200), (20, 18432, 230), (64, 100003, 100), (300, 16385, 13)])
def test_shared_coordinates(n, d, k, shared, oracle32):
    from paper_2106_05203_b200 import binding as B
    rng = np.random.default_rng(n + d)
    V = rng.standard_normal((n, d)).astype(np.float32)
    common = rng.permutation(d)[:int(shared * k)]
    V[:, common] = (20 + rng.standard_normal((n, len(common)))).astype(np.float32)
    h = B.EF21(n, d, k, 0.05)
    st = oracle_mod.State(oracle32, n, d, k, 0.05)
    h.init_grads(None, B.INIT_ZERO)
    st.init(1)
    for steps in (1, 2):
        h.step_grads(dev(V), steps)
        st.step_grads(V, steps)
        assert_state_bitwise(h, st, f"{steps} steps")
    assert h.poll() == 0

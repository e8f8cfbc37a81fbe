"""Shards between shared memory and L2 in size: the persistent kernels take their rows through a ring in shared memory."""
import numpy as np
import pytest
import torch

import ef21_inputs as inputs
from gpu_util import dev, lockstep, make_gpu, make_oracle_state

pytestmark = pytest.mark.gpu


def _workload(d, n, rows, k):
    return inputs.make_logistic("ring", n=n, d=d, N=rows, k=k, seed=d, features="bernoulli", density=0.15, gamma=0.1, T=10)


# batches of 16 rows (d <= 64) and of 8, both chunk layouts, ragged last batches, fewer batches than stages in some warps
@pytest.mark.parametrize("d,n,rows,k", [(60, 2, 17001, 1), (100, 2, 10003, 1), (123, 3, 13001, 4), (150, 2, 8005, 1), (188, 2, 7001, 16)])
def test_ring_tracks_the_oracle(d, n, rows, k, oracle32):
    from paper_2106_05203_b200 import binding as B
    w = _workload(d, n, rows, k)
    h = make_gpu(w, path=B.PATH_PERSISTENT)
    st = make_oracle_state(oracle32, w)
    h.init(B.INIT_COMPRESSED)
    st.init(0)
    lockstep(h, st, oracle32, w, 6)
    assert h.get_persistent_shape()[2] == 2 and h.get_persistent_form()[1] >= 2 and h.poll() == 0


@pytest.mark.parametrize("variant", [0, 1, 2])
@pytest.mark.parametrize("body", [1, 2])
def test_many_iterations_in_one_launch_equal_single_ones(variant, body):
    from paper_2106_05203_b200 import binding as B
    if variant == B.VARIANT_EF21_PLUS and body == 1:
        pytest.skip("the serving-warp body does not run Algorithm 3")
    w = _workload(100, 2, 10003, 2)
    states = []
    for calls in ([9], [1] * 9, [4, 5]):
        h = B.EF21(w.n, w.d, w.k, w.gamma, w.lam, total_rows=w.N)
        h.set_variant(variant)
        h.set_persistent_body(body)
        h.load_shards(dev(w.A), dev(w.y), w.row_offsets)
        h.init(B.INIT_ZERO)
        for c in calls:
            h.step(c)
        assert h.last_path == B.PATH_PERSISTENT and h.get_persistent_form()[1] >= 2 and h.poll() == 0
        states.append(h.get_state_host())
    for other in states[1:]:
        for a, b in zip(states[0], other):
            np.testing.assert_array_equal(a, b)

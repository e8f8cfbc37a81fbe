"""Persistent kernels with all workers in one cluster (messages through distributed shared memory): edges of the range of
workers, blocks and message words, and calls of many iterations against as many calls of one."""
import numpy as np
import pytest

import ef21_inputs as inputs
from gpu_util import lockstep, make_gpu, make_oracle_state

pytestmark = pytest.mark.gpu


def _workload(n, d, k, rows, seed):
    return inputs.make_logistic("one-cluster", n=n, d=d, N=n * rows + 3, k=k, seed=seed, features="bernoulli", density=0.2, gamma=0.1,
                                T=10)


# one worker, odd numbers of words, 48 words and one more, 16 blocks and one more, several blocks per worker, full d
@pytest.mark.parametrize("n,d,k,rows,one_cluster",
                         [(1, 5, 2, 9, True), (3, 128, 3, 40, True), (7, 33, 3, 20, True), (16, 64, 3, 12, True), (7, 20, 7, 12, False),
                          (17, 64, 2, 12, False), (2, 128, 24, 30, True), (2, 128, 32, 30, False), (2, 112, 1, 800, True),
                          (16, 130, 1, 20, True), (4, 127, 1, 400, True), (5, 16, 16, 10, False), (2, 100, 7, 700, True)])
def test_tracks_the_oracle(n, d, k, rows, one_cluster, oracle32):
    from paper_2106_05203_b200 import binding as B
    w = _workload(n, d, k, rows, seed=n * d + k)
    h = make_gpu(w, path=B.PATH_PERSISTENT)
    st = make_oracle_state(oracle32, w)
    h.init(B.INIT_ZERO)
    st.init(1)
    lockstep(h, st, oracle32, w, 6)
    assert h.poll() == 0
    assert h.get_persistent_form()[0] == one_cluster


@pytest.mark.parametrize("variant", [0, 1, 2])
@pytest.mark.parametrize("n,d,k,rows", [(4, 64, 4, 50), (16, 112, 1, 60), (9, 128, 7, 30), (2, 120, 2, 600)])
def test_many_iterations_are_as_many_calls(variant, n, d, k, rows):
    from paper_2106_05203_b200 import binding as B
    w = _workload(n, d, k, rows, seed=k)
    states = []
    for calls, steps in ((1, 60), (60, 1)):
        h = make_gpu(w, path=B.PATH_PERSISTENT)
        h.set_variant(variant)
        h.init(B.INIT_ZERO)
        for _ in range(calls):
            h.step(steps)
        assert h.poll() == 0 and h.last_path == B.PATH_PERSISTENT and h.get_persistent_form()[0] == (n * k <= 48)
        states.append([np.array(a) for a in h.get_state_host()])
    for a, b in zip(*states):
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32))


# both bodies (Top-1: serving warp), one and several blocks per worker, and a shape with a cluster per worker
@pytest.mark.parametrize("n,d,k,rows,one_cluster", [(4, 64, 4, 50, True), (2, 112, 1, 800, True), (16, 130, 1, 20, True), (2, 100, 7, 700, True),
                                                    (20, 112, 1, 40, False)])
def test_exchange_skeleton_has_the_form_of_the_run(n, d, k, rows, one_cluster):
    from paper_2106_05203_b200 import binding as B
    w = _workload(n, d, k, rows, seed=3)
    forms, states = [], []
    for floor in (True, False):
        h = make_gpu(w, path=B.PATH_PERSISTENT)
        h.init(B.INIT_ZERO)
        h.step(3)
        forms.append((h.get_persistent_form(), h.get_persistent_shape(), h.get_persistent_body()))
        if floor:
            h.selftest_exchange_floor(70)
            forms.append((h.get_persistent_form(), h.get_persistent_shape(), h.get_persistent_body()))
        h.step(4)                           # the skeleton leaves the state and the order of epochs alone
        assert h.poll() == 0
        states.append([np.array(a) for a in h.get_state_host()])
    assert forms[0] == forms[1] == forms[2] and forms[0][0][0] == one_cluster
    for a, b in zip(*states):
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32))

"""Persistent kernels, more than four entries of vectors wider than 128 coordinates: candidates per chunk, then one selection."""
import numpy as np
import pytest

import ef21_inputs as inputs
from gpu_util import lockstep, make_gpu, make_oracle_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,k", [(129, 5), (130, 32), (256, 6), (257, 8), (300, 16), (384, 31), (385, 5), (512, 32)])
def test_two_step_selection_tracks_the_oracle(d, k, oracle32):
    from paper_2106_05203_b200 import binding as B
    w = inputs.make_logistic("two-step", n=5, d=d, N=811, k=k, seed=d, features="bernoulli", density=0.15, gamma=0.1, T=10)
    h = make_gpu(w, path=B.PATH_PERSISTENT)
    st = make_oracle_state(oracle32, w)
    h.init(B.INIT_ZERO)               # the first messages are full of exact ties (binary features at x = 0)
    st.init(1)
    lockstep(h, st, oracle32, w, 6)
    assert h.get_persistent_body() == 2 and h.poll() == 0

"""get_state and set_state on both sides of the size where the change of layout
moves from the host to the device (api.cu)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2604_01050_gb300 import build as b
    b.build()
    import paper_2604_01050_gb300 as s
    return s


@pytest.mark.parametrize("N,P,R", [(1, 1, 1), (27, 7, 20), (115, 8, 16), (116, 8, 16), (3, 100, 36), (5, 100, 36),
                                   (290, 1, 30), (295, 1, 32), (300, 1, 32)])
def test_states_in_the_callers_layout(sb, N, P, R):
    pb = sb.create_problem_dense(np.zeros((N, N)))
    sb.set_schedule(pb, *workloads.autotune_params(R, 1), precision="fp32")
    sb.run_begin(pb, 10, P, R, seed=5)
    x, y, done = sb.get_state(pb)
    xo, yo = oracle.init_state(5, N, P, R, 0.1)
    assert done == 0 and np.array_equal(x, xo.astype(np.float32)) and np.array_equal(y, yo.astype(np.float32))
    rng = np.random.default_rng(N)
    x, y = (rng.uniform(-1, 1, (R, P, N)).astype(np.float32) for _ in range(2))
    sb.set_state(pb, x, y, 10)
    x2, y2, done = sb.get_state(pb)
    assert done == 10 and np.array_equal(x, x2) and np.array_equal(y, y2)
    sb.run_finish(pb)
    best = sb.get_best(pb)  # J = 0: every energy is 0, the first replica wins
    assert np.array_equal(best["spins"], np.where(x[:, 0] >= 0, 1, -1))

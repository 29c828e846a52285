"""Readout energies of real dense instances in fixed point on the tensor cores
(energy_fixed.cu) against the exactly rounded sums of the same terms."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2604_01050_gb300 import build as b
    b.build()
    import paper_2604_01050_gb300 as s
    return s


def _instance(kind, n, rng):
    up = np.triu(rng.standard_normal((n, n)), 1)
    h = rng.standard_normal(n)
    if kind == "tail":  # one row four orders above the others
        up[0] *= 1e4
    elif kind == "tiny":
        up, h = up * 1e-200, h * 1e-200
    elif kind == "huge":
        up, h = up * 1e200, h * 1e200
    elif kind == "field":
        up = up * 1e-9
    return up + up.T, h


@pytest.mark.parametrize("n,P,R", [(256, 1, 3), (257, 8, 17), (383, 5, 40), (640, 16, 16)])
@pytest.mark.parametrize("kind", ["gauss", "tail", "tiny", "huge", "field"])
def test_energies_are_rounded_once(sb, n, P, R, kind):
    rng = np.random.default_rng(n)
    J, h = _instance(kind, n, rng)
    pb = sb.create_problem_dense(J, h)
    sb.set_schedule(pb, precision="bf16", gamma0=4.0 * P)
    sb.run(pb, 30, P, R, seed=4)
    e, _ = sb.get_energies(pb)
    x, _, _ = sb.get_state(pb)
    best = sb.get_best(pb)
    assert np.array_equal(best["energy"], e.min(axis=1)) and np.array_equal(best["replica"], e.argmin(axis=1))
    # X = 2^k J to the nearest integer, row sums below 2^62: half a unit per term, then one rounding
    unit = 2.0 ** (math.frexp(float(np.max(np.abs(J).sum(1) + 2 * np.abs(h))))[1] - 62)
    iu = np.triu_indices(n, 1)
    for r, k in [(0, 0), (R - 1, P - 1), (R // 2, P // 2)]:
        s = np.where(x[r, k] >= 0, 1.0, -1.0)
        exact = -math.fsum(np.concatenate([J[iu] * s[iu[0]] * s[iu[1]], h * s]))
        tol = unit * 0.5 * (n * n / 2 + n) + 2.0 ** -52 * abs(exact)
        assert abs(e[r, k] - exact) <= tol, (e[r, k], exact)


def test_row_sums_past_the_fp64_range(sb):
    """No fixed point for them: the CUDA-core readout serves, as before."""
    n = 256
    J = np.zeros((n, n))
    J[0, 1:] = J[1:, 0] = 1e308
    pb = sb.create_problem_dense(J)
    sb.set_schedule(pb, precision="bf16")
    sb.run(pb, 2, 2, 2, seed=1)
    sb.get_energies(pb)

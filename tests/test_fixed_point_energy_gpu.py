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


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
@pytest.mark.parametrize("n,P,R", [(64, 4, 33), (65, 2, 70), (129, 7, 3), (256, 1, 3), (257, 8, 17), (383, 5, 40),
                                   (640, 16, 16)])
@pytest.mark.parametrize("kind", ["gauss", "tail", "tiny", "huge", "field"])
def test_energies_are_rounded_once(sb, n, P, R, kind, prec):
    rng = np.random.default_rng(n)
    J, h = _instance(kind, n, rng)
    pb = sb.create_problem_dense(J, h)
    sb.set_schedule(pb, precision=prec, gamma0=4.0 * P)
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


@pytest.mark.parametrize("n,prec", [(200, "fp32"), (300, "fp32"), (300, "bf16")])
def test_engine_and_solve_read_out_alike(sb, n, prec):
    rng = np.random.default_rng(n)
    J, h = _instance("gauss", n, rng)
    pb = sb.create_problem_dense(J, h)
    sb.set_schedule(pb, precision=prec, gamma0=32.0)
    eng = sb.engine_create(64 << 20, 4, 7)
    rid = sb.engine_submit(eng, pb, 40, 8, 5, seed=9)
    while rid not in sb.engine_step(eng):
        pass
    a = sb.engine_result(eng, rid)
    sb.run(pb, 40, 8, 5, seed=9)
    b = sb.get_best(pb)
    for k in a:
        assert np.array_equal(a[k], b[k]), k


def test_integer_couplings_beside_a_real_field(sb):
    """The e4m3 product keeps its f buffers; the spins of the readout have a buffer of their own."""
    rng = np.random.default_rng(2)
    up = np.triu(rng.integers(-3, 4, (300, 300)).astype(float), 1)
    J, h = up + up.T, rng.standard_normal(300)
    pb = sb.create_problem_dense(J, h)
    sb.set_schedule(pb, gamma0=32.0, eval_every=6)
    sb.run(pb, 31, 8, 5, seed=9)
    assert pb.info().step_kernel in (2, 5, 8, 9, 15, 16)
    e, _ = sb.get_energies(pb)
    x, _, _ = sb.get_state(pb)
    s = np.where(x >= 0, 1.0, -1.0)
    ref = -0.5 * np.einsum("rki,ij,rkj->rk", s, J, s) - s @ h
    assert np.allclose(e, ref, rtol=1e-12, atol=0)


def test_row_sums_past_the_fp64_range(sb):
    """No fixed point for them: the CUDA-core readout serves, as before."""
    n = 256
    J = np.zeros((n, n))
    J[0, 1:] = J[1:, 0] = 1e308
    pb = sb.create_problem_dense(J)
    sb.set_schedule(pb, precision="bf16")
    sb.run(pb, 2, 2, 2, seed=1)
    sb.get_energies(pb)

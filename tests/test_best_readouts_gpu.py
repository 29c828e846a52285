"""The best spins of a run over several readouts, some of them at the same
step: they keep the energy reported beside them, on both sides of the size
where their copy is a kernel of its own (init_readout.cu)."""
import numpy as np
import pytest

from sbqa_cases import create, regular

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2604_01050_gb300 import build as b
    b.build()
    import paper_2604_01050_gb300 as s
    return s


def _energies(spec, spins):
    _, n, rp, col, val, h = spec
    rows = np.repeat(np.arange(n), np.diff(rp))
    s = spins.astype(np.float64)
    return -0.5 * (s[:, rows] * s[:, col] * val).sum(1) - (0.0 if h is None else s @ h)


def _instance(n, integer):
    _, spec = regular(n, 4, n)
    if integer:
        spec = (*spec[:4], np.where(spec[4] > 0, 1.0, -1.0), None)
    return spec


@pytest.mark.parametrize("n", [16383, 16384, 16641])
@pytest.mark.parametrize("integer", [False, True])
@pytest.mark.parametrize("again", ["finish", "rewind"])
def test_a_worse_readout_at_the_same_step_keeps_the_best(sb, n, integer, again):
    """A good state is read out, then a random one at the same step: by a second finish, or by going
    back past a readout of eval_every.  dt is so small that a state keeps its signs."""
    spec = _instance(n, integer)
    P, R, S = 4, 3, 4
    pb = create(sb, spec)
    sb.set_schedule(pb, precision="fp32", gamma0=16.0, eval_every=2 if again == "rewind" else 0)
    sb.run(pb, 120, P, R, seed=1)
    x, _, _ = sb.get_state(pb)
    good = np.where(x >= 0, 0.5, -0.5).astype(np.float32)
    bad = np.random.default_rng(n).choice(np.float32([-0.5, 0.5]), size=x.shape)
    zero = np.zeros_like(x)
    sb.set_schedule(pb, precision="fp32", dt=1e-4, eval_every=2 if again == "rewind" else 0)
    sb.run_begin(pb, S, P, R, seed=2)
    for state in (good, bad):
        if again == "finish":
            sb.set_state(pb, state, zero, S)
            sb.run_finish(pb)
        else:
            sb.set_state(pb, state, zero, 0)
            sb.run_advance(pb, 2)
    if again == "rewind":
        sb.run_advance(pb, S)
        sb.run_finish(pb)
    best = sb.get_best(pb)
    want = _energies(spec, np.where(good > 0, 1, -1).reshape(R * P, n)).reshape(R, P)
    assert np.allclose(best["energy"], want.min(axis=1), rtol=1e-10)
    assert np.allclose(_energies(spec, best["spins"]), best["energy"], rtol=1e-10)
    assert np.array_equal(best["replica"], want.argmin(axis=1))
    assert np.all(best["step"] == (S - 1 if again == "finish" else 1))

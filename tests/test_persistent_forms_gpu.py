"""The persistent CSR forms that small instances do not take by themselves:
the streaming solvers, which the host-side hook SBQA_TEST_PERSIST_PASSES=0
sends every run batch to, against the per-step kernels, bit for bit; and the
bounded waits of every form (SBQA_TEST_SKIP_BARRIER_STEP=n keeps block 0 from
publishing step n), which end with a status and leave the handle usable."""
import numpy as np
import pytest

import workloads
from sbqa_cases import create, lattice, regular

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2604_01050_gb300 import build as b
    b.build()
    import paper_2604_01050_gb300 as s
    return s


def _solve(sb, spec, P, R, steps, ks, pb=None, **kw):
    pb = pb or create(sb, spec)
    sb.set_schedule(pb, *workloads.autotune_params(R, 2), kernel_select=ks, **kw)
    sb.run(pb, steps, P, R, seed=11)
    return pb


def _equal(sb, a, b):
    for u, v in zip(sb.get_state(a)[:2], sb.get_state(b)[:2]):
        assert np.array_equal(u, v)
    ea, eb = sb.get_best(a), sb.get_best(b)
    for k in ea:
        assert np.array_equal(ea[k], eb[k]), k
    assert np.array_equal(sb.get_energies(a)[0], sb.get_energies(b)[0])


# instance, P, R, precision
CASES = {
    "one_item": (lambda: lattice(5, 1), 8, 2, "auto"),         # one block of columns, fewer items than warps
    "p1_ragged": (lambda: lattice(6, 2), 1, 5, "auto"),
    "p2_ragged": (lambda: regular(700, 6, 2), 2, 67, "fp32"),  # lanes cut by R * P
    "ring3": (lambda: lattice(9, 3), 3, 40, "auto"),           # a ring with padding columns
    "ring100": (lambda: regular(900, 6, 3), 100, 2, "bf16"),
    "several_items": (lambda: lattice(20, 4), 32, 16, "auto"),
    "degree8": (lambda: regular(5000, 7, 6), 16, 8, "fp32"),   # the generator's rows are of the degree or one off it
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("variant", ["threshold", "ballistic"])
def test_streaming_equals_per_step(sb, monkeypatch, name, variant):
    make, P, R, prec = CASES[name]
    _, spec = make()
    kw = dict(precision=prec, variant=variant, gamma0=4.0 * P, eval_every=13)
    a = _solve(sb, spec, P, R, 41, 1, **kw)
    monkeypatch.setenv("SBQA_TEST_PERSIST_PASSES", "0")
    b = _solve(sb, spec, P, R, 41, 2, **kw)
    assert a.info().step_kernel == (6 if variant == "ballistic" else 0)
    assert b.info().step_kernel == (14 if variant == "ballistic" else 4)
    _equal(sb, a, b)


# instance, variant, whether the streaming form
WAITS = {
    "short lists": (lambda: regular(3000, 6, 7), "threshold", False),
    "long lists": (lambda: regular(3000, 12, 7), "threshold", False),
    "ballistic": (lambda: regular(3000, 6, 7), "ballistic", False),
    "streaming": (lambda: regular(3000, 6, 7), "threshold", True),
    "streaming ballistic": (lambda: regular(3000, 6, 7), "ballistic", True),
}


@pytest.mark.parametrize("name", sorted(WAITS))
def test_a_wait_that_runs_out_is_reported_and_the_handle_recovers(sb, monkeypatch, name):
    make, variant, streaming = WAITS[name]
    _, spec = make()
    kw = dict(precision="fp32", variant=variant, gamma0=32.0)
    if streaming:
        monkeypatch.setenv("SBQA_TEST_PERSIST_PASSES", "0")
    monkeypatch.setenv("SBQA_TEST_SKIP_BARRIER_STEP", "10")
    pb = _solve(sb, spec, 8, 16, 40, 2, **kw)
    assert pb.info().step_kernel == (14 if variant == "ballistic" else 4)
    with pytest.raises(sb.SBQAError) as e:
        sb.get_best(pb)
    assert e.value.status == sb.ERR_TIMEOUT
    monkeypatch.delenv("SBQA_TEST_SKIP_BARRIER_STEP")
    _solve(sb, spec, 8, 16, 40, 2, pb=pb, **kw)
    _equal(sb, _solve(sb, spec, 8, 16, 40, 1, **kw), pb)


@pytest.mark.parametrize("L,P,R", [(14, 16, 64), (14, 7, 128), (16, 16, 128), (20, 8, 48)])
def test_the_ballistic_form_the_autotuner_keeps(sb, L, P, R):
    """Shapes where it times the on-chip form and the streaming one."""
    _, spec = lattice(L, 3)
    kw = dict(variant="ballistic", gamma0=4.0 * P, eval_every=13)
    a, b = (_solve(sb, spec, P, R, 30, ks, **kw) for ks in (1, 0))
    assert b.info().step_kernel == 14 and 0 < b.info().persistent_ms < b.info().variant_ms[0]
    _equal(sb, a, b)


@pytest.mark.parametrize("value", [2.5, -7.0, np.inf, np.nan])
def test_streaming_takes_states_from_outside_the_wall(sb, monkeypatch, value):
    """The streaming ballistic solver has no bit to spare in a position: it takes any state, as the
    per-step kernel does."""
    _, spec = lattice(6, 8)
    P, R, steps = 4, 8, 12
    monkeypatch.setenv("SBQA_TEST_PERSIST_PASSES", "0")
    out = []
    for ks in (1, 2):
        pb = create(sb, spec)
        sb.set_schedule(pb, *workloads.autotune_params(R, 2), kernel_select=ks, variant="ballistic", gamma0=16.0)
        sb.run_begin(pb, steps, P, R, seed=3)
        x, y, _ = sb.get_state(pb)
        x[1, 2, 5] = value
        sb.set_state(pb, x, y, 0)
        sb.run_advance(pb, steps)
        assert pb.info().step_kernel == (14 if ks == 2 else 6)
        out.append(sb.get_state(pb))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])

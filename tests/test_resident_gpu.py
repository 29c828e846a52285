"""The persistent CSR solvers with the state on the chip (solve_persistent.cu)
against the per-step kernels, bit for bit: items of 128 and 256 columns, state
in tensor memory, in shared memory and in global memory, ragged columns and
rings, runs in several launches; and the forms that take another kernel."""
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


def _run(sb, spec, P, R, steps, ks, **kw):
    pb = create(sb, spec)
    sb.set_schedule(pb, *workloads.autotune_params(R, 2), kernel_select=ks, **kw)
    sb.run(pb, steps, P, R, seed=11)
    x, y, _ = sb.get_state(pb)
    return pb, x, y, sb.get_best(pb), sb.get_energies(pb)


# instance, P, R, precision: the passes of a warp (24 warps on 152 SMs) in the comment
CASES = {
    "one_item": (lambda: lattice(5, 1), 8, 2, "auto"),               # fewer items than warps, C < 128
    "p1_ragged": (lambda: lattice(6, 2), 1, 5, "auto"),              # one column per run, 5 of 8 in a lane
    "p2_ragged": (lambda: regular(700, 6, 2), 2, 67, "fp32"),        # lanes cut by C, 256 columns
    "ring3": (lambda: lattice(9, 3), 3, 40, "auto"),                 # general ring, padding columns
    "ring100": (lambda: regular(900, 6, 3), 100, 2, "bf16"),         # a ring over 16 lanes
    "tmem": (lambda: lattice(20, 4), 32, 16, "auto"),                # 5 passes
    "slot": (lambda: regular(42000, 6, 4), 8, 16, "bf16"),           # 6 passes of two items
    "global": (lambda: lattice(20, 5), 32, 32, "auto"),              # 9 passes
    "global_real": (lambda: regular(30000, 4, 5), 16, 16, "fp32"),   # 9 passes, 4 slots
    "degree8": (lambda: regular(5000, 8, 6), 16, 8, "fp32"),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("variant", ["threshold", "ballistic"])
def test_resident_equals_per_step(sb, name, variant):
    make, P, R, prec = CASES[name]
    _, spec = make()
    kw = dict(precision=prec, variant=variant, gamma0=4.0 * P, eval_every=13)
    a = _run(sb, spec, P, R, 41, 1, **kw)
    b = _run(sb, spec, P, R, 41, 2, **kw)
    assert a[0].info().step_kernel == (6 if variant == "ballistic" else 0)
    assert b[0].info().step_kernel == (14 if variant == "ballistic" else 4)
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
    for k in a[3]:
        assert np.array_equal(a[3][k], b[3][k]), k
    assert np.array_equal(a[4][0], b[4][0]) and np.array_equal(a[4][1], b[4][1])


def _signs(spec):
    kind, n, rp, col, val, _ = spec
    return kind, n, rp, col, np.where(val > 0, 1.0, -1.0), None


@pytest.mark.parametrize("degree", [9, 12, 13, 17, 24, 25, 31, 32])
@pytest.mark.parametrize("values,P,R", [("pm1", 8, 16), ("pm1", 12, 10), ("fp32", 16, 16), ("bf16", 4, 9)])
def test_long_lists_equal_per_step(sb, degree, values, P, R):
    """Rows of 9 to 32 entries, in groups of 12 slots with remainders, on half and whole warps, several
    passes a warp for the first shape.  (The generator's rows are of the degree or one off it; past 32
    entries the per-step kernels serve.)"""
    _, spec = regular(9000 if (values, P) == ("pm1", 8) else 1200, degree, degree)
    if values == "pm1":
        spec = _signs(spec)
    prec = "auto" if values == "pm1" else values
    kw = dict(precision=prec, gamma0=4.0 * P, eval_every=17)
    a = _run(sb, spec, P, R, 40, 1, **kw)
    b = _run(sb, spec, P, R, 40, 2, **kw)
    longest = int(np.diff(spec[2]).max())
    assert a[0].info().step_kernel == 0 and b[0].info().step_kernel == (4 if longest <= 32 else 0)
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
    for k in a[3]:
        assert np.array_equal(a[3][k], b[3][k]), k


@pytest.mark.parametrize("degree,variant,want", [(35, "threshold", 0), (9, "ballistic", 6)])
def test_degrees_past_the_lists_stay_per_step(sb, degree, variant, want):
    _, spec = regular(1200, degree, 5)
    assert _run(sb, spec, 8, 16, 10, 2, variant=variant)[0].info().step_kernel == want


@pytest.mark.parametrize("variant", ["threshold", "ballistic"])
@pytest.mark.parametrize("cut", [1, 2, 3, 18])
def test_stretches_and_restarts(sb, variant, cut):
    """Launches that begin at odd and even steps, and a restart two steps back: no code or position of
    an earlier launch is taken for a new one."""
    _, spec = regular(3000, 6, 7)
    P, R, steps = 8, 16, 20
    kw = dict(variant=variant, gamma0=32.0, precision="fp32")
    _, x, y, _, _ = _run(sb, spec, P, R, steps, 1, **kw)
    pb = create(sb, spec)
    sb.set_schedule(pb, *workloads.autotune_params(R, 2), kernel_select=2, **kw)
    sb.run_begin(pb, steps, P, R, seed=11)
    sb.run_advance(pb, cut)
    xc, yc, done = sb.get_state(pb)
    sb.run_advance(pb, 2)
    sb.set_state(pb, xc, yc, done)
    sb.run_advance(pb, 1)
    sb.run_advance(pb, steps)
    x2, y2, _ = sb.get_state(pb)
    assert np.array_equal(x, x2) and np.array_equal(y, y2)


@pytest.mark.parametrize("value", [2.5, -7.0, np.inf, np.nan])
def test_ballistic_states_from_outside_the_wall(sb, value):
    """Positions of magnitude 2 and more use the bit that tells steps apart: such a run stays on the
    per-step kernel and equals it."""
    _, spec = lattice(6, 8)
    P, R, steps = 4, 8, 12
    out = []
    for ks in (1, 2):
        pb = create(sb, spec)
        sb.set_schedule(pb, *workloads.autotune_params(R, 2), kernel_select=ks, variant="ballistic", gamma0=16.0)
        sb.run_begin(pb, steps, P, R, seed=3)
        x, y, _ = sb.get_state(pb)
        x[1, 2, 5] = value
        sb.set_state(pb, x, y, 0)
        sb.run_advance(pb, steps)
        assert pb.info().step_kernel == 6
        out.append(sb.get_state(pb))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("N,P,R", [(1, 1, 1), (31, 3, 5), (33, 7, 9), (216, 12, 3), (1000, 64, 2)])
def test_state_round_trip(sb, N, P, R):
    """get_state and set_state in the caller's layout: what goes in comes out, padding untouched."""
    J = np.zeros((N, N))
    pb = sb.create_problem_dense(J)
    sb.set_schedule(pb, *workloads.autotune_params(R, 1))
    sb.run_begin(pb, 10, P, R, seed=5)
    rng = np.random.default_rng(N)
    x, y = (rng.uniform(-1, 1, (R, P, N)).astype(np.float32) for _ in range(2))
    sb.set_state(pb, x, y, 4)
    x2, y2, done = sb.get_state(pb)
    assert done == 4 and np.array_equal(x, x2) and np.array_equal(y, y2)

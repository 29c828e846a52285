"""Handles on a device without the memory for a request: the host-side test
hook SBQA_TEST_FAIL_ALLOC=bytes:count makes the library's next `count` requests
of at least `bytes` bytes fail as on a full device."""
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


def _gauss(sb, n, **kw):
    up = np.triu(np.random.default_rng(n).standard_normal((n, n)), 1)
    pb = sb.create_problem_dense(up + up.T)
    sb.set_schedule(pb, precision="fp32", **kw)
    return pb


def test_a_handle_whose_results_did_not_fit(sb, monkeypatch):
    """Same columns, more runs: only the block of the results (200 KB) has to grow, and does not get the
    memory.  The handle has no results then, synchronises, and solves once there is memory again.
    (Integer couplings: no planes to give up for it.)"""
    up = np.triu(np.random.default_rng(1).integers(-3, 4, (200, 200)).astype(float), 1)
    pb, fresh = (sb.create_problem_dense(up + up.T) for _ in range(2))
    sb.set_schedule(pb)
    sb.set_schedule(fresh)
    sb.run(pb, 2, 128, 8, seed=1)
    monkeypatch.setenv("SBQA_TEST_FAIL_ALLOC", "100000:1")
    with pytest.raises(sb.SBQAError) as e:
        sb.run(pb, 2, 1, 1000, seed=2)
    assert e.value.status == sb.ERR_OOM
    monkeypatch.delenv("SBQA_TEST_FAIL_ALLOC")
    sb.synchronize(pb)
    with pytest.raises(sb.SBQAError) as e:
        sb.get_best(pb)
    assert e.value.status == sb.ERR_STATE
    sb.run(pb, 2, 1, 1000, seed=2)
    sb.run(fresh, 2, 1, 1000, seed=2)
    a, b = sb.get_best(pb), sb.get_best(fresh)
    for k in a:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("failures", ["6500000:1", "2000000:1"])
def test_the_readout_planes_keep_no_run_out(sb, monkeypatch, failures):
    """The planes of the fixed-point readout (6.6 MB) do not fit, or a larger run (2.6 MB of positions)
    does not fit beside them: the FP64 readout serves, to the same spins."""
    fresh = _gauss(sb, 640, gamma0=32.0)
    sb.run(fresh, 30, 8, 128, seed=2)
    a, ea = sb.get_best(fresh), sb.get_energies(fresh)[0]
    pb = _gauss(sb, 640, gamma0=32.0)
    if failures.startswith("2"):
        sb.run(pb, 30, 8, 4, seed=1)
    monkeypatch.setenv("SBQA_TEST_FAIL_ALLOC", failures)
    for again in range(2):  # the second time the kept graph
        sb.run(pb, 30, 8, 128, seed=2)
        b, eb = sb.get_best(pb), sb.get_energies(pb)[0]
        assert np.array_equal(a["spins"], b["spins"]) and np.array_equal(a["replica"], b["replica"])
        assert np.allclose(ea, eb, rtol=1e-12, atol=1e-9) and not np.array_equal(ea, eb)


def test_a_run_that_does_not_fit_without_the_planes_either(sb, monkeypatch):
    pb = _gauss(sb, 640, gamma0=32.0)
    sb.run(pb, 30, 8, 4, seed=1)
    monkeypatch.setenv("SBQA_TEST_FAIL_ALLOC", "2000001:2")
    with pytest.raises(sb.SBQAError) as e:
        sb.run(pb, 30, 8, 128, seed=2)
    assert e.value.status == sb.ERR_OOM
    sb.run(pb, 30, 8, 128, seed=2)
    assert np.isfinite(sb.get_best(pb)["energy"]).all()


@pytest.mark.parametrize("N,P,R", [(1, 1, 20000), (3, 7, 1500), (33, 12, 60), (500, 3, 50)])
@pytest.mark.parametrize("variant", ["threshold", "ballistic"])
def test_state_transfers_without_a_slice(sb, monkeypatch, N, P, R, variant):
    """No memory for the slice that state transfers pass through: get_state and set_state work as before,
    in several slices, and the run goes on the same way; a state outside the wall is still seen."""
    up = np.triu(np.random.default_rng(N).standard_normal((N, N)), 1)
    J = up + up.T
    rows, cols = np.nonzero(J)
    if variant == "ballistic":  # sparse, a ring, for the form that looks at the state's range
        rows = np.repeat(np.arange(N), 2) if N > 2 else np.zeros(0, int)
        cols = np.sort(np.stack([np.arange(N) - 1, np.arange(N) + 1], 1) % N, axis=1).ravel() if N > 2 else rows
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=N))])
    val = np.ones(rows.size) if variant == "ballistic" else J[rows, cols]
    out = []
    for fail in (False, True):
        pb = sb.create_problem_csr(N, rp, cols, val)
        sb.set_schedule(pb, precision="fp32", variant=variant, gamma0=4.0 * P, kernel_select=2)
        sb.run_begin(pb, 12, P, R, seed=3)
        sb.run_advance(pb, 5)
        if fail:
            monkeypatch.setenv("SBQA_TEST_FAIL_ALLOC", "1:1000")
        x, y, done = sb.get_state(pb)
        x[R - 1, P - 1, N - 1] = 2.5
        y[0, 0, 0] = -3.0
        sb.set_state(pb, x, y, done)
        x2, y2, _ = sb.get_state(pb)
        assert np.array_equal(x, x2) and np.array_equal(y, y2)
        kernel = pb.info().step_kernel
        monkeypatch.delenv("SBQA_TEST_FAIL_ALLOC", raising=False)
        sb.run_advance(pb, 7)
        sb.run_finish(pb)
        out.append((x, y, kernel, *sb.get_state(pb)[:2], sb.get_best(pb)["spins"]))
    assert all(np.array_equal(a, b) for a, b in zip(*out))
    if variant == "ballistic":
        assert out[0][2] == 6


def test_the_kept_graph_after_the_planes_were_given_up(sb, monkeypatch):
    """A run of the other form asks for buffers of its own and does not get them, with the planes or
    without; no buffer of the first form has moved.  Its kept graph names the planes and is not used."""
    pb = _gauss(sb, 640, gamma0=32.0)
    sb.run(pb, 30, 8, 16, seed=2)
    a, ea = sb.get_best(pb), sb.get_energies(pb)[0]
    sb.set_schedule(pb, precision="fp32", gamma0=32.0, variant="ballistic")
    monkeypatch.setenv("SBQA_TEST_FAIL_ALLOC", "100:2")
    with pytest.raises(sb.SBQAError) as e:
        sb.run(pb, 30, 8, 16, seed=2)
    assert e.value.status == sb.ERR_OOM
    monkeypatch.delenv("SBQA_TEST_FAIL_ALLOC")
    sb.set_schedule(pb, precision="fp32", gamma0=32.0)
    sb.run(pb, 30, 8, 16, seed=2)
    b, eb = sb.get_best(pb), sb.get_energies(pb)[0]
    assert np.array_equal(a["spins"], b["spins"])
    assert np.allclose(ea, eb, rtol=1e-12, atol=1e-9) and not np.array_equal(ea, eb)

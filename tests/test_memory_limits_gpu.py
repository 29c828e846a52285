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
    """Same columns, more runs: only the block of the results (300 KB) has to grow, and does not get the
    memory.  The handle has no results then, synchronises, and solves once there is memory again."""
    pb = _gauss(sb, 300)
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
    fresh = _gauss(sb, 300)
    sb.run(fresh, 2, 1, 1000, seed=2)
    a, b = sb.get_best(pb), sb.get_best(fresh)
    for k in a:
        assert np.array_equal(a[k], b[k]), k

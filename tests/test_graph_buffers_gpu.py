"""The kept graph of a solve against buffers that have moved since (api.cu)."""
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


def test_a_solve_after_a_larger_run_uses_its_own_buffers(sb):
    """run_begin with one run more moves some of the buffers (the readout's spins, 64 -> 96 KiB) and not
    others, which stay within their size classes.  A second handle takes the spins' old block for its
    positions; the solve that comes back to the first shape must not write there."""
    rng = np.random.default_rng(65)
    up = np.triu(rng.standard_normal((65, 65)), 1)
    pb = sb.create_problem_dense(up + up.T)
    sb.set_schedule(pb, precision="fp32")
    sb.release_cached_memory()
    sb.run(pb, 100, 1, 256, seed=3)
    first, e_first = sb.get_best(pb), sb.get_energies(pb)[0]
    sb.run_begin(pb, 100, 1, 257, seed=4)
    other = sb.create_problem_dense(np.zeros((32, 32)))
    sb.set_schedule(other)
    sb.run_begin(other, 10, 1, 512, seed=5)  # 32 x 512 floats: 64 KiB
    before = sb.get_state(other)
    sb.run(pb, 100, 1, 256, seed=3)
    again, e_again = sb.get_best(pb), sb.get_energies(pb)[0]
    after = sb.get_state(other)
    assert np.array_equal(before[0], after[0]) and np.array_equal(before[1], after[1])
    assert np.array_equal(e_first, e_again)
    for k in first:
        assert np.array_equal(first[k], again[k]), k


def test_a_solve_after_another_operand_form(sb):
    """e4m3, then a bfloat16 run_begin that needs larger operand buffers, then e4m3 again."""
    rng = np.random.default_rng(2)
    up = np.triu(rng.integers(-9, 10, (300, 300)).astype(float), 1)
    pb = sb.create_problem_dense(up + up.T)
    sb.set_schedule(pb, gamma0=32.0, kernel_select=1)
    sb.run(pb, 40, 8, 16, seed=3)
    first = sb.get_best(pb)
    sb.set_schedule(pb, gamma0=32.0, kernel_select=1, precision="bf16")
    sb.run_begin(pb, 40, 8, 16, seed=3)
    sb.set_schedule(pb, gamma0=32.0, kernel_select=1)
    sb.run(pb, 40, 8, 16, seed=3)
    again = sb.get_best(pb)
    for k in first:
        assert np.array_equal(first[k], again[k]), k


def test_schedule_tables_that_came_back_to_their_old_block(sb, monkeypatch):
    """A run that does not get memory for larger tables leaves the handle without them; another handle
    uses their old block and returns it.  The first shape's tables lie there again, and are made again."""
    rng = np.random.default_rng(40)
    up = np.triu(rng.standard_normal((40, 40)), 1)
    pb, other = (sb.create_problem_dense(up + up.T) for _ in range(2))
    sb.set_schedule(pb, precision="fp32", gamma0=1.0)
    sb.set_schedule(other, precision="fp32", gamma0=30.0)
    sb.release_cached_memory()
    sb.run(pb, 1000, 1, 250, seed=3)  # tables of 1000 x 250 entries: 1 MB
    first = sb.get_best(pb)
    monkeypatch.setenv("SBQA_TEST_FAIL_ALLOC", "1150000:1")
    with pytest.raises(sb.SBQAError):
        sb.run(pb, 1000, 1, 300, seed=3)
    monkeypatch.delenv("SBQA_TEST_FAIL_ALLOC")
    sb.run(other, 1000, 1, 250, seed=3)
    sb.get_best(other)
    other.destroy()
    sb.run(pb, 1000, 1, 250, seed=3)
    again = sb.get_best(pb)
    for k in first:
        assert np.array_equal(first[k], again[k]), k

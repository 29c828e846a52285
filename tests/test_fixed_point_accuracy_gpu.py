"""Readout energies of real dense instances are no further from the exact ones
than the FP64 sums of the CUDA-core kernel, whatever the ranges of J and h: the
fixed-point form serves where that holds and the FP64 kernel elsewhere
(energy_fixed.cu)."""
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


def _instance(kind, n):
    rng = np.random.default_rng(n)
    up, h = np.triu(rng.standard_normal((n, n)), 1), np.zeros(n)
    if kind == "fields":  # of the size of the coupling sums
        h = rng.standard_normal(n) * np.sqrt(n)
    elif kind == "large fields":
        h = rng.standard_normal(n) * n
    elif kind == "field only":
        up, h = up * 1e-9, rng.standard_normal(n)
    elif kind.startswith("pinned"):
        h = rng.standard_normal(n)
        h[0] = float(kind.split()[1])
    elif kind == "opposed":
        h = rng.standard_normal(n)
        h[0], h[1] = 1e30, -1e30
    elif kind == "row":
        up[0] *= 1e4
    elif kind == "pairs":
        up[0, 1], up[2, 3] = 1e30, -1e30
    elif kind == "sparse rows":  # most spins neither coupled nor in a field
        up[:, n // 4:] = 0
    return up + up.T, h


def _fp64_order(J, h, S):
    """The sums of k_energy_dense: rows in entry order, four rows a warp, eight warps a block, blocks over
    lanes, a shuffle tree.  S [n][columns]."""
    n, C = S.shape
    t = np.zeros((n, C))
    for j in range(n):
        t += J[:, j, None] * S[j]
    v = S * (0.5 * t + h[:, None])
    blocks = -(-n // 32)
    v = np.concatenate([v, np.zeros((blocks * 32 - n, C))]).reshape(blocks, 8, 4, C)
    part = np.zeros((blocks, C))
    warps = np.zeros((blocks, 8, C))
    for a in range(4):
        warps += v[:, :, a]
    for w in range(8):
        part += warps[:, w]
    lanes = np.zeros((32, C))
    for k in range(blocks):
        lanes[k % 32] += part[k]
    for o in (16, 8, 4, 2, 1):
        lanes[:o] += lanes[o:2 * o]
    return -lanes[0]


def _two_sum(a, b):
    s = a + b
    z = s - a
    return s, (a - (s - z)) + (b - z)


def _exact(J, h, S):
    """(hi, lo) of the energies with about 100 bits."""
    hi, lo = np.zeros(S.shape), np.zeros(S.shape)
    for j in range(S.shape[0]):
        hi, e = _two_sum(hi, 0.5 * J[:, j, None] * S[j])
        lo = lo + e
    hi, e = _two_sum(hi, np.broadcast_to(h[:, None], S.shape))
    lo = lo + e
    eh, el = np.zeros(S.shape[1]), np.zeros(S.shape[1])
    for i in range(S.shape[0]):
        eh, e = _two_sum(eh, -S[i] * hi[i])
        el = el + (e - S[i] * lo[i])
    return eh, el


# instance, whether the fixed point serves
CASES = [("gauss", 64, True), ("gauss", 300, True), ("gauss", 1024, True), ("gauss", 2048, True),
         ("fields", 64, True), ("fields", 1024, True), ("large fields", 300, True), ("large fields", 1024, True),
         ("field only", 300, True), ("row", 64, True), ("row", 300, False), ("row", 1024, False),
         ("pinned 1e6", 300, False), ("pinned 1e9", 2048, False), ("pinned 1e12", 64, False),
         ("opposed", 300, False), ("pairs", 300, False), ("sparse rows", 300, True)]


def _spins(J, h, count):
    """[n][count] random spins; in the second half of the columns half of the rows are then aligned."""
    rng = np.random.default_rng(7)
    S = rng.choice([-1.0, 1.0], size=(len(h), count))
    for i in range(len(h)):
        free = np.arange(count) >= count // 2
        free &= rng.random(count) < 0.5
        S[i, free] = np.where(J[i] @ S[:, free] + h[i] >= 0, 1.0, -1.0)
    return S


def _read_out(sb, J, h, prec, S, P):
    """The energies a run reports that ends in the spins S."""
    n, C = S.shape
    pb = sb.create_problem_dense(J, h)
    sb.set_schedule(pb, precision=prec)
    sb.run_begin(pb, 4, P, C // P, seed=1)
    x = np.ascontiguousarray(0.5 * S.T, dtype=np.float32).reshape(C // P, P, n)
    sb.set_state(pb, x, np.zeros_like(x), 4)
    sb.run_finish(pb)
    return sb.get_energies(pb)[0].reshape(-1)


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
@pytest.mark.parametrize("kind,n,fixed", CASES)
def test_no_further_off_than_fp64_sums(sb, kind, n, fixed, prec):
    """Over 128 configurations: root mean square of the distance from the exact energies, up to the
    10 % that two such samples may differ by.  Where the FP64 kernel serves, its very sums."""
    J, h = _instance(kind, n)
    S = _spins(J, h, 128)
    e = _read_out(sb, J, h, prec, S, 8)
    ref = _fp64_order(J, h, S)
    eh, el = _exact(J, h, S)
    rms = lambda v: np.sqrt(np.mean(((v - eh) - el) ** 2))  # noqa: E731
    assert np.array_equal(e, ref) != fixed
    assert rms(e) <= 1.1 * rms(ref), (rms(e), rms(ref))


def test_sums_past_the_fp64_range(sb):
    """|J| row sums overflow: no fixed point, and the FP64 sums as they come, infinite ones included."""
    n = 256
    J = _instance("gauss", n)[0] * 1e300
    J[0, 1], J[0, 2] = 1e308, -1e308
    J[1, 0], J[2, 0] = J[0, 1], J[0, 2]
    S = np.random.default_rng(3).choice([-1.0, 1.0], size=(n, 128))
    e = _read_out(sb, J, np.zeros(n), "bf16", S, 4)
    with np.errstate(over="ignore", invalid="ignore"):
        ref = _fp64_order(J, np.zeros(n), S)
    assert np.isfinite(ref).any() and np.isinf(ref).any()
    assert np.array_equal(e, ref)

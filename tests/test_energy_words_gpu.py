"""sbqa_energies_csr_noalloc where spins are read as words (integer J, aligned
rows, whole chunks of 128 configurations) and a byte at a time: the same
energies from both, and the exact ones."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("n,count", [(33, 128), (19500, 128), (2601, 1024), (2600, 1022), (700, 4000)])
def test_words_equal_bytes(n, count, real):
    import torch

    from paper_2604_01050_gb300 import build as b
    b.build()
    import paper_2604_01050_gb300 as sb
    n, rp, col, val, _ = workloads.random_regular(n, 6, n, 0.0)
    val = val if real else np.rint(10 * val)
    spins = np.random.default_rng(count).choice(np.array([-1, 1], dtype=np.int8), size=(n, count))
    dev = torch.device("cuda")
    a_rp = torch.from_numpy(rp.astype(np.int32)).to(dev)
    a_col = torch.from_numpy(col.astype(np.int32)).to(dev)
    a_val = torch.from_numpy(val if real else val.astype(np.int32)).to(dev)
    out = []
    for ld in (-(-count // 4) * 4, -(-count // 4) * 4 + 1):  # rows on 4-byte boundaries, and not
        s = torch.zeros((n, ld), dtype=torch.int8, device=dev)
        s[:, :count] = torch.from_numpy(spins).to(dev)
        e = torch.zeros(count, dtype=torch.float64, device=dev)
        torch.cuda.synchronize()
        sb.energies_csr_noalloc(n, a_rp.data_ptr(), a_col.data_ptr(), s.data_ptr(), ld, count, energy=e.data_ptr(),
                                **{"val_f64" if real else "val_i32": a_val.data_ptr()})
        torch.cuda.synchronize()
        out.append(e.cpu().numpy())
    assert np.array_equal(out[0], out[1])
    rows = np.repeat(np.arange(n), np.diff(rp))
    k = count - 1
    ref = -0.5 * np.sum(val * spins[rows, k] * spins[col, k].astype(float))
    assert abs(out[0][k] - ref) <= (1e-12 * np.abs(val).sum() if real else 0.0)

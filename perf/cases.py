"""Performance cases of the SBQA solver: what its users run, over the range of sizes they run it at.

Every case goes through the public entry points of ``paper_2604_01050_gb300`` (the ctypes binding
of ``include/sbqa.h``) with host arrays in and out.  Five kinds of use:

  solve       a handle with its schedule is kept; one pass solves it and fetches the best spins of
              every run and the energies of all replicas
  create      one pass takes an instance from the caller's arrays to its best spins: create the
              problem, set the schedule, solve, fetch, destroy
  checkpoint  one pass advances a run part of the way, fetches its state, hands that state to
              another handle and finishes there
  serve       one pass sends a mix of requests through the batching engine in a closed loop
  energies    one pass evaluates caller-supplied spin configurations on the device

Instance families: dense Sherrington-Kirkpatrick with +-1 couplings ("sk") or Gaussian ones
("gauss"), the periodic cubic lattice with +-1 bonds ("lattice"; n is L^3), and random graphs of a
given degree with Gaussian couplings and fields ("graph").
"""
import numpy as np
import torch

import paper_2604_01050_gb300 as sb


def _case(use, family, n, P, R, steps, **more):
    c = {"use": use, "family": family, "n": n, "degree": 0, "P": P, "R": R, "steps": steps, "precision": "auto",
         "variant": "threshold", "eval_every": 0, "gamma0": 1.0}
    c.update(more)
    return c


def listed():
    return [
        # a small fully connected instance, many times over: launch and step latency
        {"name": "sk64", **_case("solve", "sk", 64, 8, 16, 1000)},
        # a mid-size dense instance with real couplings at the default (FP32) precision
        {"name": "gauss1000", **_case("solve", "gauss", 1000, 16, 16, 100)},
        # the dense tensor-core workload with exact integer couplings
        {"name": "sk2000", **_case("solve", "sk", 2000, 32, 32, 500)},
        # dense Gaussian couplings in bfloat16, keeping the best of several readouts along the anneal
        {"name": "gauss2000_bf16_readouts", **_case("solve", "gauss", 2000, 32, 32, 300, precision="bf16",
                                                    eval_every=100)},
        # a small 3D spin glass, the size of a time-to-target study
        {"name": "lattice10", **_case("solve", "lattice", 1000, 16, 64, 500)},
        # the 3D spin-glass benchmark: many runs of many replicas
        {"name": "lattice16", **_case("solve", "lattice", 4096, 32, 64, 500)},
        # the large sparse benchmark: 100 000 spins, fields, bfloat16 couplings
        {"name": "graph1e5_bf16", **_case("solve", "graph", 100000, 16, 8, 200, degree=6, precision="bf16")},
        # a ragged mid-size sparse instance of the degree of annealer hardware graphs: odd sizes, FP32
        # couplings, a replica count that is no power of two
        {"name": "graph3001_d20", **_case("solve", "graph", 3001, 12, 10, 300, degree=20)},
        # the ballistic form with a checkpoint and a resume on another handle
        {"name": "lattice12_ballistic_resume", **_case("checkpoint", "lattice", 1728, 16, 32, 200,
                                                       variant="ballistic", gamma0=64.0)},
        # a new dense instance from host arrays to its best spins, once
        {"name": "create_sk1024", **_case("create", "sk", 1024, 16, 16, 100)},
        # a request mix of dense and lattice instances through the batching engine
        {"name": "serve8", **_case("serve", "mix", 3000, 0, 16, 200, requests=8)},
        # energies of given spin configurations from device arrays
        {"name": "energies_lattice16", **_case("energies", "lattice", 4096, 1, 2048, 0)},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.randrange(8)
    P = rng.choice([1, 4, 7, 8, 12, 16, 24, 32, 64])
    R = _log_int(rng, 1, 40)
    steps = _log_int(rng, 40, 300)
    if kind == 0:  # small dense, integer or real
        return _case("solve", rng.choice(["sk", "gauss"]), _log_int(rng, 24, 250), P, R, _log_int(rng, 100, 1000))
    if kind == 1:  # dense real couplings at the default precision
        return _case("solve", "gauss", _log_int(rng, 256, 1500), P, max(1, min(R, 512 // P)), _log_int(rng, 20, 100))
    if kind == 2:  # dense tensor cores, with or without readouts along the way
        fam = rng.choice(["sk", "gauss"])
        return _case("solve", fam, _log_int(rng, 300, 2300), P, max(1, min(R, 1024 // P)), steps,
                     precision="auto" if fam == "sk" else "bf16", eval_every=rng.choice([0, 0, 100]))
    if kind == 3:  # lattices
        L = rng.randrange(4, 21)
        return _case("solve", "lattice", L ** 3, P, max(1, min(R, 1024 // P)), steps)
    if kind == 4:  # sparse graphs
        return _case("solve", "graph", _log_int(rng, 300, 60000), P, max(1, min(R, 128 // P)), steps,
                     degree=rng.choice([4, 6, 8, 12, 16, 20]), precision=rng.choice(["auto", "bf16"]))
    if kind == 5:
        L = rng.randrange(4, 15)
        return _case("checkpoint", "lattice", L ** 3, P, max(1, min(R, 512 // P)), 2 * _log_int(rng, 20, 100),
                     variant=rng.choice(["ballistic", "threshold"]), gamma0=4.0 * P)
    if kind == 6:
        return _case("create", rng.choice(["sk", "gauss"]), _log_int(rng, 64, 2000), min(P, 32), min(R, 16),
                     _log_int(rng, 50, 200), precision="bf16" if rng.random() < 0.5 else "auto")
    if rng.random() < 0.5:
        return _case("serve", "mix", _log_int(rng, 300, 3000), 0, 16, 200, requests=rng.randrange(4, 9))
    return _case("energies", "lattice", rng.randrange(4, 17) ** 3, 1, _log_int(rng, 1, 2048), 0)


# ---------------------------------------------------------------- instances
def _dense(family, n, rng):
    if family == "sk":
        a = np.triu(rng.integers(0, 2, size=(n, n), dtype=np.int8) * 2 - 1, k=1)
        return (a + a.T).astype(np.float64)
    a = np.triu(rng.standard_normal((n, n)), k=1)
    return a + a.T


def _csr(n, i, j, w):
    """Symmetric CSR of the distinct undirected edges (i, j) with weights w."""
    lo, hi = np.minimum(i, j), np.maximum(i, j)
    _, first = np.unique(lo * n + hi, return_index=True)
    i, j, w = lo[first], hi[first], w[first]
    rows, cols, vals = np.concatenate([i, j]), np.concatenate([j, i]), np.concatenate([w, w])
    order = np.argsort(rows * n + cols)
    row_ptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(rows, minlength=n), out=row_ptr[1:])
    return row_ptr, cols[order].astype(np.int32), vals[order].astype(np.float64)


def _sparse(family, n, degree, rng):
    """(row_ptr, col, val, h) of a periodic cubic lattice of n = L^3 spins, or of a random graph made
    of degree / 2 random cycles over n spins (an edge drawn twice counts once)."""
    if family == "lattice":
        L = int(round(n ** (1.0 / 3.0)))
        s = np.arange(n, dtype=np.int64)
        x, y, z = s % L, (s // L) % L, s // (L * L)
        j = np.concatenate([(x + 1) % L + L * y + L * L * z, x + L * ((y + 1) % L) + L * L * z,
                            x + L * y + L * L * ((z + 1) % L)])
        return *_csr(n, np.tile(s, 3), j, rng.choice([-1.0, 1.0], size=3 * n)), None
    i, j = [], []
    for _ in range(degree // 2):
        p = rng.permutation(n)
        i.append(p)
        j.append(np.roll(p, 1))
    return *_csr(n, np.concatenate(i), np.concatenate(j), rng.standard_normal(n * (degree // 2))), \
        0.1 * rng.standard_normal(n)


def _instance(case, rng):
    if case["family"] in ("sk", "gauss"):
        return {"J": _dense(case["family"], case["n"], rng)}
    rp, col, val, h = _sparse(case["family"], case["n"], case["degree"], rng)
    return {"rp": rp, "col": col, "val": val, "h": h}


def _create(inst):
    if "J" in inst:
        return sb.create_problem_dense(inst["J"])
    return sb.create_problem_csr(inst["rp"].size - 1, inst["rp"], inst["col"], inst["val"], inst["h"])


def _schedule(pb, case, s):
    sb.set_schedule(pb, s["beta"], s["alpha"], precision=case["precision"], variant=case["variant"],
                    eval_every=case["eval_every"], gamma0=case["gamma0"])


def prepare(case, seed):
    rng = np.random.default_rng([seed, 17])
    s = {"case": case, "seed": int(rng.integers(1 << 62)), "beta": rng.uniform(0.5, 1.5, case["R"]),
         "alpha": rng.uniform(0.5, 1.0, case["R"])}
    if case["use"] == "serve":
        # a server's problem library: a third of the pool's instances are lattices, sizes spread over the range
        pool = []
        for k in range(6):
            n = int(round(64 * (case["n"] / 64.0) ** (k / 5.0)))
            if k % 3 == 2:
                L = max(3, int(round(n ** (1.0 / 3.0))))
                inst = dict(zip(("rp", "col", "val", "h"), _sparse("lattice", L ** 3, 0, rng)))
            else:
                inst = {"J": _dense("sk", n, rng)}
            pb = _create(inst)
            _schedule(pb, case, s)
            pool.append(pb)
        s["requests"] = [(pool[q % 6], int(rng.choice([8, 16, 32])), int(rng.integers(1 << 62)))
                         for q in range(case["requests"])]
        s["engine"] = sb.engine_create(2 << 30, 16, 100)
        return s
    inst = _instance(case, rng)
    if case["use"] == "energies":
        dev = torch.device("cuda")
        n, count = case["n"], case["R"]
        s["row_ptr"] = torch.from_numpy(inst["rp"].astype(np.int32)).to(dev)
        s["col"] = torch.from_numpy(inst["col"]).to(dev)
        s["val"] = torch.from_numpy(inst["val"].astype(np.int32)).to(dev)
        s["spins"] = torch.from_numpy(rng.integers(0, 2, size=(n, count), dtype=np.int8) * 2 - 1).to(dev)
        s["e_int"] = torch.zeros(count, dtype=torch.int64, device=dev)
        s["e"] = torch.zeros(count, dtype=torch.float64, device=dev)
        return s
    if case["use"] == "create":
        s["inst"] = inst
        return s
    s["pb"] = _create(inst)
    _schedule(s["pb"], case, s)
    if case["use"] == "checkpoint":
        s["resumed"] = _create(inst)
        _schedule(s["resumed"], case, s)
    return s


def _solve(pb, case, s):
    sb.run(pb, case["steps"], case["P"], case["R"], s["seed"])
    return {"best": sb.get_best(pb), "energies": sb.get_energies(pb)}


def run(s):
    case = s["case"]
    if case["use"] == "solve":
        return _solve(s["pb"], case, s)
    if case["use"] == "create":
        pb = _create(s["inst"])
        _schedule(pb, case, s)
        out = _solve(pb, case, s)
        pb.destroy()
        return out
    if case["use"] == "checkpoint":
        S, P, R = case["steps"], case["P"], case["R"]
        sb.run_begin(s["pb"], S, P, R, s["seed"])
        sb.run_advance(s["pb"], S // 2)
        x, y, done = sb.get_state(s["pb"])
        sb.run_begin(s["resumed"], S, P, R, s["seed"])
        sb.set_state(s["resumed"], x, y, done)
        sb.run_advance(s["resumed"], S - done)
        sb.run_finish(s["resumed"])
        return {"x": x, "y": y, "best": sb.get_best(s["resumed"])}
    if case["use"] == "serve":
        eng = s["engine"]
        ids = [sb.engine_submit(eng, pb, case["steps"], P, case["R"], seed) for pb, P, seed in s["requests"]]
        left = set(ids)
        while left:
            left.difference_update(sb.engine_step(eng))
        return [sb.engine_result(eng, rid) for rid in ids]
    sb.energies_csr_noalloc(case["n"], s["row_ptr"].data_ptr(), s["col"].data_ptr(), s["spins"].data_ptr(), case["R"],
                            case["R"], val_i32=s["val"].data_ptr(), energy_int=s["e_int"].data_ptr(),
                            energy=s["e"].data_ptr(), stream=torch.cuda.current_stream())
    return s["e_int"], s["e"]


def work(case):
    """Couplings read once, results written once (the state never has to leave the chip), and the
    arithmetic of the steps: one multiply-add per coupling and about 14 operations per replica-spin."""
    n, P, R, S = case["n"], case["P"], case["R"], case["steps"]
    if case["use"] == "serve":
        nbytes = flops = 0.0
        for q in range(case["requests"]):
            m = int(round(64 * (n / 64.0) ** ((q % 6) / 5.0)))
            lattice = q % 6 % 3 == 2
            m = max(3, int(round(m ** (1.0 / 3.0)))) ** 3 if lattice else m
            nnz = 6 * m if lattice else m * m
            nbytes += nnz + R * m
            flops += (2.0 * nnz + 14.0 * m) * 16 * R * S  # 16: the middle replica count
        return {"bytes": nbytes, "flops": flops}
    nnz = n * n if case["family"] in ("sk", "gauss") else n * (6 if case["family"] == "lattice" else case["degree"])
    if case["use"] == "energies":
        return {"bytes": n * R + 8.0 * nnz + 16.0 * R, "flops": 2.0 * nnz * R}
    C = P * R
    # bytes of a coupling: sparse ones carry their column; a new dense instance arrives in FP64
    per = 8 if case["family"] in ("lattice", "graph") or case["use"] == "create" else \
        {"sk": 1, "gauss": 2 if case["precision"] == "bf16" else 4}[case["family"]]
    readouts = 1 + ((S - 1) // case["eval_every"] if case["eval_every"] else 0)
    state = 16.0 * n * C if case["use"] == "checkpoint" else 0.0
    return {"bytes": float(per) * nnz + R * n + 16.0 * C + state,
            "flops": (2.0 * nnz + 14.0 * n) * C * S + 2.0 * nnz * C * readouts}


# ---------------------------------------------------------------- 64-bit values
def _uniform(seed, ctr, amp):
    """SplitMix64 output number ctr of the seed, its top 24 bits mapped to [-amp, amp)."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (ctr + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    m = (z >> np.uint64(40)).astype(np.int64) - (1 << 23)
    return (m.astype(np.float32) * np.float32(2.0 ** -23) * np.float32(amp)).astype(np.float64)


def exact(case, seed):
    """The states of a ballistic checkpoint and the energies of given configurations have 64-bit
    values; a thresholded anneal is chaotic, so its spins have none."""
    if case["use"] == "energies":
        s = prepare(case, seed)
        rows = torch.repeat_interleave(torch.arange(case["n"], device=s["col"].device),
                                       (s["row_ptr"][1:] - s["row_ptr"][:-1]).long())
        e = torch.zeros(case["R"], dtype=torch.float64, device=s["col"].device)
        for a in range(0, rows.numel(), 4096):
            r, c = rows[a:a + 4096], s["col"][a:a + 4096].long()
            e -= 0.5 * (s["val"][a:a + 4096, None].double() * s["spins"][r].double() * s["spins"][c].double()).sum(0)
        return None, e
    if case["use"] != "checkpoint" or case["variant"] != "ballistic":
        return None
    rng = np.random.default_rng([seed, 17])
    run_seed = int(rng.integers(1 << 62))
    P, R, S, n = case["P"], case["R"], case["steps"], case["n"]
    beta, alpha = rng.uniform(0.5, 1.5, R), rng.uniform(0.5, 1.0, R)
    inst = _instance(case, rng)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    J = torch.sparse_csr_tensor(torch.from_numpy(inst["rp"]), torch.from_numpy(inst["col"].astype(np.int64)),
                                torch.from_numpy(inst["val"]), size=(n, n)).to(dev)
    el = np.arange(R * P * n, dtype=np.uint64)
    x, y = (torch.from_numpy(_uniform(run_seed, 2 * el + np.uint64(w), 0.1).reshape(R, P, n)).to(dev) for w in (0, 1))
    c0 = 0.5 * np.sqrt(n / float((inst["val"] ** 2).sum()))
    dt = 0.5
    for k in range(S // 2):
        tau = k / S
        gam = case["gamma0"] * ((1 - tau) ** alpha + 1e-5)
        jp = torch.from_numpy(-np.log(np.tanh(beta * gam / P)) / (2 * beta)).to(dev)[:, None, None]
        G = (J @ x.reshape(R * P, n).T).T.reshape(R, P, n)
        y = y + dt * (-(1.0 - tau) / P * x + c0 / P * G + jp * (x.roll(1, 1) + x.roll(-1, 1)))
        x = x + dt / P * y
        wall = x.abs() > 1
        x = torch.where(wall, x.sign(), x)
        y = torch.where(wall, torch.zeros_like(y), y)
    return {"x": x, "y": y, "best": None}

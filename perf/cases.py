"""The calls whose speed a user of this package feels, as cases for a timing harness.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)`` one more of the
same ranges; ``prepare(case, seed)`` makes what a program has in hand before the call (the instance
of a tensor it described, or the device cores it wants checked), ``run(state)`` is one pass through
the public entry points, ``work(case)`` what the pass cannot do without, and ``exact(case, seed)``
the same outputs from plain numpy in 64 bits where they do not hang on the order of roundings.

Kinds of pass:
  cross    an adaptive TT cross: ``TTCross.run``, then its ranks and every core on the device
  batch    several tensors of uneven shape in one launch: ``run_batch``, then every core
  rebuild  the cores rebuilt from the pivots of an earlier run: ``TTCross.rebuild_cores``
  error    the relative error of given device cores: ``sampled_error_noalloc``
The cores of a tensor go one after the other into a device buffer that the program keeps, as large
as the ranks may get (what is behind the last core stays zero).

The tensors are functions of their indices.  What the seed decides: the sizes of a Hilbert
tensor's modes (a little under the case's n, every mode of a ragged case, else the last one), the
amplitudes of the Maxwellians, the weights of the caller's function, the TT cores, and the error
samples everywhere.
"""
import random

import numpy as np
import torch

from paper_2407_11290_gb300 import ttcross

GOOD = (ttcross.OK, ttcross.NOT_CONVERGED)
MASK = (1 << 64) - 1


def _case(name, kind, tensor, d, n, eps, cap, rank, samples=10**6, **more):
    """``rank``: about the rank the bonds reach; ``ranks``: prescribed ranks, as a text."""
    c = dict(name=name, kind=kind, tensor=tensor, d=d, n=n, eps=eps, cap=cap, rank=rank,
             samples=samples, pieces=0, residual="recompute", precision="fp64", ragged=False,
             ranks="", grid="", screen=0, count=1)
    c.update(more)
    return c


def listed():
    return [
        # the smallest tensor of the repository's workloads, checked on every entry: a call whose
        # latency counts (an inner step of a program that compresses many small tensors)
        _case("cross_hilbert3d_n32", "cross", "hilbert", 3, 32, 1e-10, 64, 13, samples=0, pieces=1,
              ragged=True),
        # the ordinary 6D workload in the library's default form (every residual formed afresh)
        _case("cross_hilbert6d_n64", "cross", "hilbert", 6, 64, 1e-8, 64, 15, pieces=2),
        # the benchmark's tensor in its headline form: stored residuals, FP64
        _case("cross_hilbert6d_n256_stored", "cross", "hilbert", 6, 256, 1e-10, 128, 23, pieces=4,
              residual="stored"),
        # the same size in the mixed form, every mode of a size of its own
        _case("cross_hilbert6d_n256_mixed", "cross", "hilbert", 6, 256, 1e-10, 128, 23, pieces=4,
              residual="stored", precision="split", ragged=True),
        # the 3x+3v Maxwellian to 1e-6 at rank cap 256, the largest single run: high ranks
        _case("cross_maxwellian6d_n64", "cross", "maxwellian", 6, 64, 1e-6, 256, 150,
              residual="stored"),
        # the 2d2v distribution at its published size and prescribed ranks: wide superblocks
        _case("cross_2d2v_n1000", "cross", "xv", 4, 1000, 0.0, 20, 12, ranks="10,5,20",
              grid="1,8,8,1", residual="stored"),
        # a TT of known ranks found again from its entries (recompression), default form
        _case("cross_tt5d_n48", "cross", "tt", 5, 48, 1e-8, 16, 8, samples=10**5),
        # a function of the caller's, evaluated through the batch callback
        _case("cross_user4d_n64", "cross", "user", 4, 64, 1e-7, 40, 16, residual="stored"),
        # a superblock too large to look through: a random sample set with row / column refinement
        _case("cross_sampled6d_n256", "cross", "hilbert", 6, 256, 0.0, 24, 24, screen=2**18),
        # many tensors of uneven shape in one launch, the mixed form: the batch workload's recipe
        _case("batch_maxwellian_x12", "batch", "maxwellian", 0, 0, 1e-6, 64, 55, residual="stored",
              precision="split", count=12),
        # the cores built again from the pivot sets, as after loading them from a file
        _case("rebuild_hilbert6d_n300", "rebuild", "hilbert", 6, 300, 0.0, 18, 17,
              ranks="15,17,18,17,15", grid="1,2,4,4,2,1", residual="stored"),
        # the check of a TT that another program holds on the device
        _case("error_hilbert6d_n64", "error", "hilbert", 6, 64, 0.0, 16, 16),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["small", "cross", "cross", "stored", "stored", "mixed", "maxwellian", "xv",
                       "tt", "user", "sampled", "batch", "rebuild", "error"])
    if kind == "small":
        n, e = _log_int(rng, 12, 72), rng.choice([6, 8, 10])
        return _drawn("cross", "hilbert", rng.choice([2, 3]), n, 10.0**-e, 64, _hilbert_rank(3, n, e),
                      samples=0, ragged=True, residual=rng.choice(["recompute", "stored"]))
    if kind in ("cross", "stored", "mixed"):
        d, e = rng.choice([4, 5, 6]), rng.choice([6, 8, 10])
        n = _log_int(rng, 20, 256 if kind != "cross" else 160)
        more = {} if kind == "cross" else {"residual": "stored"}
        if kind == "mixed":
            more["precision"] = "split"
        return _drawn("cross", "hilbert", d, n, 10.0**-e, 64, _hilbert_rank(d, n, e),
                      pieces=rng.choice([0, 1, 2, 4]), ragged=rng.random() < 0.5,
                      samples=_log_int(rng, 20000, 10**6), **more)
    if kind == "maxwellian":
        d = rng.choice([4, 5, 6])
        return _drawn("cross", "maxwellian", d, _log_int(rng, 24, 96), 10.0**-rng.choice([3, 4, 6]),
                      rng.choice([32, 64, 96]), 50, residual="stored",
                      precision=rng.choice(["fp64", "split"]),
                      samples=_log_int(rng, 20000, 10**6))
    if kind == "xv":
        D = rng.choice([2, 3])
        n = _log_int(rng, 60, 600 if D == 2 else 400)
        rk = [rng.randint(4, 20) for _ in range(2 * D - 1)]
        return _drawn("cross", "xv", 2 * D, n, 0.0, max(rk), 12, ranks=",".join(map(str, rk)),
                      residual=rng.choice(["recompute", "stored"]) if n < 150 else "stored")
    if kind == "tt":
        return _drawn("cross", "tt", rng.choice([3, 4, 5]), _log_int(rng, 12, 64), 1e-8, 16,
                      rng.randint(2, 10), samples=_log_int(rng, 10000, 10**5),
                      residual=rng.choice(["recompute", "stored"]))
    if kind == "user":
        return _drawn("cross", "user", rng.choice([3, 4, 5]), _log_int(rng, 16, 96),
                      10.0**-rng.choice([5, 6, 7]), 40, 14, samples=_log_int(rng, 20000, 10**6),
                      residual=rng.choice(["recompute", "stored"]))
    if kind == "sampled":
        cap = _log_int(rng, 6, 24)
        return _drawn("cross", "hilbert", rng.choice([4, 5, 6]), _log_int(rng, 48, 300), 0.0, cap,
                      cap, screen=2 ** rng.randint(10, 18))
    if kind == "batch":
        return _drawn("batch", "maxwellian", 0, 0, 1e-6, rng.choice([24, 32, 48]), 40,
                      residual="stored", precision=rng.choice(["fp64", "split"]),
                      count=rng.randint(2, 8), samples=_log_int(rng, 20000, 10**6))
    if kind == "rebuild":
        d, n = rng.choice([3, 4, 5, 6]), _log_int(rng, 32, 300)
        r = rng.randint(6, _hilbert_rank(d, n, 10))
        return _drawn("rebuild", "hilbert", d, n, 0.0, r, r, residual="stored",
                      ragged=rng.random() < 0.5)
    d, r = rng.choice([4, 5, 6]), rng.randint(6, 48)
    return _drawn("error", "hilbert", d, _log_int(rng, 16, 256), 0.0, r, r,
                  samples=_log_int(rng, 20000, 10**6), ragged=rng.random() < 0.5)


def _drawn(*args, **more):
    c = _case("", *args, **more)
    del c["name"]
    return c


def _hilbert_rank(d, n, e):
    return max(2, round(0.32 * e * float(np.log(d * n))))


# ---------------------------------------------------------------------------
# inputs


def _rng(case, seed):
    return random.Random(f"{case['kind']} {case['tensor']} {case['d']} {case['n']} {seed}")


def _numbers(text, count, other):
    return [int(v) for v in text.split(",")] if text else [other] * count


def _sizes(case, seed):
    """The mode sizes."""
    d, n = case["d"], case["n"]
    if case["tensor"] == "xv":
        return [2 * n, n] * (d // 2)
    ns = [n] * d
    if case["tensor"] == "hilbert":
        rng = _rng(case, 1)
        ns[-1] = n - seed % max(2, n // 8)  # another size for each of a few seeds in a row
        if case["ragged"]:
            ns[:-1] = [n - (rng.randrange(n) + 3 * seed * (m + 1)) % max(2, n // 8)
                       for m in range(d - 1)]
    return ns


def _tt_cores(case, seed):
    """TT cores with Gaussian entries, scaled so that entries stay about 1."""
    g = np.random.default_rng([seed, case["d"], case["n"]])
    r = [1] + [case["rank"]] * (case["d"] - 1) + [1]
    r = [min(a, case["n"]) for a in r]
    cores = [g.standard_normal((r[m], case["n"], r[m + 1])) / np.sqrt(r[m])
             for m in range(case["d"])]
    for c in cores:
        c[:, 0, :] = np.abs(c[:, 0, :]) + 0.5
    return r, cores


def _maxwellian(rng, dx, dv, spread):
    a = [spread * rng.random() for _ in range(3)] if spread else [
        0.5 + 0.05 * (rng.random() - 0.5), 0.3 + 0.03 * (rng.random() - 0.5),
        0.2 + 0.02 * (rng.random() - 0.5)]
    return {"kind": "maxwellian", "dx": dx, "dv": dv, "a_rho": a[0], "a_u": a[1], "a_T": a[2],
            "vmin": -8.0, "vmax": 8.0}


def _weights(ns, rng):
    return [(0.5 + rng.random()) / (n - 1) ** 2 for n in ns]


def _user_function(ns, rng):
    """1 / sqrt(0.1 + sum_m w_m i_m^2), a few torch operations per call."""
    w = _weights(ns, rng)

    def fn(idx, out):
        out.fill_(0.1)
        for m, wm in enumerate(w):
            i = idx[:, m].to(torch.float64)
            out.addcmul_(i, i, value=wm)
        out.rsqrt_()

    return {"kind": "user", "fn": fn}


def _instance(case, seed, ns, gen):
    more = {}
    if case["ranks"]:
        more["bond_max_rank"] = _numbers(case["ranks"], 0, 0)
    if case["screen"]:
        more.update(screen_samples=case["screen"], screen_seed=seed + 1, rook_rounds=4)
    return ttcross.TTCross(ns, gen, max_rank=case["cap"], nsamples=case["samples"], seed=seed + 5,
                           residual=case["residual"], precision=case["precision"], **more)


def _generator(case, seed, ns):
    rng, tensor, d = _rng(case, seed), case["tensor"], case["d"]
    if tensor == "maxwellian":
        return _maxwellian(rng, d // 2, d - d // 2, 0.0)
    if tensor == "xv":
        return {"kind": "maxwellian_xv", "dx": d // 2, "dv": d // 2,
                "a_rho": 0.875 - 0.05 * rng.random(), "a_T": 0.4 - 0.05 * rng.random(),
                "a_u": 0.75 - 0.05 * rng.random(), "vmin": -3.0, "vmax": 3.0}
    if tensor == "tt":
        r, cores = _tt_cores(case, seed)
        return {"kind": "tt", "ranks": r, "cores": cores}
    if tensor == "user":
        return _user_function(ns, rng)
    return {"kind": "hilbert"}


def _batch(case, seed):
    """Shapes of the batch recipe (d = 4, 5, 6 in turn, n from 32 to 128), amplitudes U(0, 0.5)."""
    rng, ws = _rng(case, seed), []
    for i in range(case["count"]):
        d, n = 4 + i % 3, (64, 32, 96, 48, 128, 32, 64, 48, 32, 96, 64, 48)[i % 12]
        ws.append(([n] * d, _maxwellian(rng, d // 2, d - d // 2, 0.5)))
    return ws


def _error_cores(case, seed, ns):
    """Cores a program wants checked against 1 / (1 + i_1 + ... + i_d): the exponential sum
    sum_j w_j prod_m exp(-t_j i_m) of 1/x, x in [1, 1 + sum (n_m - 1)] (trapezoidal rule in log t),
    with a random orthogonal change of basis on every bond.  Returns (w, t, cores)."""
    r = case["rank"]
    top = float(sum(ns))
    u = np.linspace(np.log(1e-3 / top), np.log(8.0), r)
    t = np.exp(u)
    w = (u[1] - u[0]) * t * np.exp(-t)
    g = np.random.default_rng([seed, r])
    qs = [np.linalg.qr(g.standard_normal((r, r)))[0] for _ in range(len(ns) - 1)]
    cores = []
    for m, n in enumerate(ns):
        f = np.exp(-np.outer(np.arange(n), t))  # [n, r]
        if m == 0:
            c = (f * w) @ qs[0]
            c = c[None]
        elif m == len(ns) - 1:
            c = (qs[-1].T @ f.T)[:, :, None]
        else:
            c = np.einsum("jp,ij,jq->piq", qs[m - 1], f, qs[m], optimize=True)
        cores.append(np.ascontiguousarray(c))
    return w, t, cores


def _room(case, d, n):
    """Values of the cores of a d-mode tensor at the largest ranks they may get."""
    r = min(case["cap"], 2 * case["rank"] + 8)
    return 2 * n * r + (d - 2) * r * n * r


def _buffer(case, d, n):
    return torch.zeros(_room(case, d, n), dtype=torch.float64, device="cuda")


def prepare(case, seed):
    s = {"case": case, "seed": seed}
    if case["kind"] == "batch":
        ws = _batch(case, seed)
        s["crosses"] = [_instance(case, seed + i, ns, gen) for i, (ns, gen) in enumerate(ws)]
        s["buffers"] = [_buffer(case, len(ns), max(ns)) for ns, _ in ws]
        return s
    ns = _sizes(case, seed)
    if case["kind"] == "error":
        s["n"] = ns
        s["cores"] = [torch.from_numpy(c).cuda() for c in _error_cores(case, seed, ns)[2]]
        s["out"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        return s
    s["grid"] = None
    if case["grid"] or case["pieces"]:
        s["grid"] = _numbers(case["grid"], case["d"], case["pieces"])
    s["cross"] = _instance(case, seed, ns, _generator(case, seed, ns))
    s["buffer"] = _buffer(case, case["d"], 2 * case["n"] if case["tensor"] == "xv" else case["n"])
    if case["kind"] == "rebuild":
        s["cross"].run(case["eps"], subtensor_grid=s["grid"])
        s["cross"].sync(allow=GOOD)
    return s


# ---------------------------------------------------------------------------
# one pass


def _result(c, buffer):
    at = 0
    for k in range(1, c.d + 1):
        core = c.core(k, device=True)
        buffer[at:at + core.numel()].copy_(core.view(-1))
        at += core.numel()
    return {"ranks": c.ranks(), "cores": buffer}


def run(s):
    case = s["case"]
    if case["kind"] == "error":
        ttcross.sampled_error_noalloc(s["n"], {"kind": "hilbert"}, s["cores"], case["samples"],
                                      s["seed"] + 5, s["out"])
        return {"err": s["out"]}
    if case["kind"] == "batch":
        ttcross.run_batch(s["crosses"], case["eps"])
        for c in s["crosses"]:
            c.sync(allow=GOOD)
        return [_result(c, b) for c, b in zip(s["crosses"], s["buffers"])]
    c = s["cross"]
    if case["kind"] == "rebuild":
        c.rebuild_cores()
    else:
        c.run(case["eps"], subtensor_grid=s["grid"])
        c.sync(allow=GOOD)
    return _result(c, s["buffer"])


# ---------------------------------------------------------------------------
# what a pass cannot do without


def _tensor_work(case, ns, ranks):
    """Every entry of the final superblocks formed and compared once (a residual at half the final
    rank), the error samples through the cores, the cores written."""
    d = len(ns)
    r = [1] + ranks + [1]
    out = sum(r[m] * ns[m] * r[m + 1] for m in range(d))
    ns_err = case["samples"] if case["samples"] > 0 else int(np.prod([float(n) for n in ns]))
    ns_err = min(float(ns_err), float(np.prod([float(n) for n in ns])))
    if case["kind"] == "rebuild":
        return 8.0 * out, 2.0 * sum(r[m] * ns[m] * r[m + 1] ** 2 for m in range(d - 1))
    if case["screen"]:
        flops = sum(float(case["screen"]) * r[b + 1] ** 2 for b in range(d - 1))
    else:
        flops = sum(float(r[b] * ns[b]) * (ns[b + 1] * r[b + 2]) * r[b + 1] for b in range(d - 1))
    return 8.0 * out, flops + 2.0 * ns_err * max(a * b for a, b in zip(r, r[1:]))


def work(case):
    if case["kind"] == "error":
        r, d, n = case["rank"], case["d"], case["n"]
        return {"bytes": 8.0 * (2 * n * r + (d - 2) * n * r * r),
                "flops": 2.0 * case["samples"] * ((d - 2) * r * r + r)}
    if case["kind"] == "batch":
        got = [_tensor_work(case, ns, [min(case["rank"], ns[0])] * (len(ns) - 1))
               for ns, _ in _batch(case, 0)]
    else:
        ranks = _numbers(case["ranks"], case["d"] - 1, case["rank"])
        got = [_tensor_work(case, _sizes(case, 0), ranks)]
    return {"bytes": sum(b for b, _ in got), "flops": sum(f for _, f in got)}


# ---------------------------------------------------------------------------
# the same in plain numpy


def _mix(seed, k):
    """Outputs k (an array) of SplitMix64 started with ``seed``."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed & MASK) + (k + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _samples(ns, count, seed):
    """The error's sample indices [count, d]: floor(x n / 2^64), sample-major."""
    total = int(np.prod([float(n) for n in ns]))
    d = len(ns)
    if count <= 0 or count >= total:
        l = np.arange(total)
        out = np.empty((total, d), np.int64)
        for m, n in enumerate(ns):
            out[:, m] = l % n
            l //= n
        return out
    x = _mix(seed, np.arange(count * d, dtype=np.uint64)).reshape(count, d)
    hi, lo = x >> np.uint64(32), x & np.uint64(0xFFFFFFFF)
    n = np.asarray(ns, np.uint64)
    return ((hi * n + ((lo * n) >> np.uint64(32))) >> np.uint64(32)).astype(np.int64)


def _tt_entries(cores, idx):
    """Entries of a TT at idx [count, d], a block of samples at a time."""
    out = np.empty(len(idx))
    for i in range(0, len(idx), 1 << 15):
        j = idx[i:i + (1 << 15)]
        v = cores[0][0, j[:, 0], :]
        for m in range(1, len(cores)):
            v = np.einsum("sp,psq->sq", v, cores[m][:, j[:, m], :])
        out[i:i + len(j)] = v[:, 0]
    return out


def _grid(rows, n, m, cols):
    """Multi-indices [len(rows) n, m len(cols), d] of a superblock: row p n + i, column q m + j."""
    rows, cols = np.asarray(rows, np.int64), np.asarray(cols, np.int64)
    a = np.concatenate([np.repeat(rows, n, axis=0), np.tile(np.arange(n), len(rows))[:, None]], 1)
    c = np.concatenate([np.tile(np.arange(m), len(cols))[:, None], np.repeat(cols, m, axis=0)], 1)
    shape = (len(a), len(c))
    return np.concatenate([np.broadcast_to(a[:, None], shape + a.shape[1:]),
                           np.broadcast_to(c[None], shape + c.shape[1:])], 2)


def _numpy_cross(case, seed, ns, entries):
    """The adaptive cross by its definition, its tensor without ties between residuals: every bond
    takes the entry of largest residual of its superblock, all bonds at once, while it is above
    tau rms(X); when none is, the sampled error ends the run or tau goes down tenfold."""
    d, eps = len(ns), case["eps"]
    idx = _samples(ns, case["samples"], seed + 5)
    x = entries(idx)
    rms, x0 = np.sqrt(np.mean(x ** 2)), entries(np.zeros((1, d), np.int64))[0]
    start = tuple(idx[np.argmax(np.abs(x))]) if np.abs(x).max() > abs(x0) else (0,) * d
    left = [[()]] + [[start[:b + 1]] for b in range(d - 1)]   # left[b]: I of the modes < b
    right = [[start[b:]] for b in range(1, d)] + [[()]]       # right[b]: J of the modes > b
    blocks = [entries(_grid(left[b], ns[b], ns[b + 1], right[b + 1])) for b in range(d - 1)]

    def factors(b):  # pivot columns and rows of bond b's superblock, and their common entries
        rows = [left[b].index(i[:-1]) * ns[b] + int(i[-1]) for i in left[b + 1]]
        cols = [right[b + 1].index(j[1:]) * ns[b + 1] + int(j[0]) for j in right[b]]
        return blocks[b][:, cols], blocks[b][rows], blocks[b][np.ix_(rows, cols)]

    def cores():
        out = []
        for b in range(d - 1):
            c, r, p = factors(b)
            out.append(np.linalg.solve(p.T, c.T).T.reshape(len(left[b]), ns[b], -1))
        return out + [r[:, :, None]]

    tau = eps
    for _ in range(1000):
        found = []
        for b in range(d - 1):
            c, r, p = factors(b)
            e = blocks[b] - c @ np.linalg.solve(p, r)
            row, col = divmod(int(np.argmax(np.abs(e))), e.shape[1])
            add = abs(e[row, col]) > tau * rms and len(right[b]) < case["cap"]
            found.append((add, left[b][row // ns[b]] + (row % ns[b],),
                          (col % ns[b + 1],) + right[b + 1][col // ns[b + 1]]))
        if not any(f[0] for f in found):
            err = np.linalg.norm(x - _tt_entries(cores(), idx)) / np.linalg.norm(x)
            if err <= eps or tau < 0.5e-6 * eps:
                break
            tau /= 10
        for b, (add, i, j) in enumerate(found):
            if add:
                left[b + 1].append(i)
                right[b].append(j)
        for b in range(d - 1):
            blocks[b] = entries(_grid(left[b], ns[b], ns[b + 1], right[b + 1]))
    return cores()


def _entries(case, seed, ns):
    """The tensor of a case as a function of multi-indices [..., d], where no two of its residuals
    tie up to rounding; else None."""
    if case["tensor"] == "tt":
        g = _tt_cores(case, seed)[1]
        return lambda idx: _tt_entries(g, idx.reshape(-1, len(ns))).reshape(idx.shape[:-1])
    if case["tensor"] == "user":
        w = _weights(ns, _rng(case, seed))

        def value(idx):
            out = np.full(idx.shape[:-1], 0.1)
            for m, wm in enumerate(w):
                out += idx[..., m].astype(np.float64) ** 2 * wm
            return 1.0 / np.sqrt(out)
        return value
    return None


def exact(case, seed):
    if case["kind"] == "error":
        ns = _sizes(case, seed)
        w, t, _ = _error_cores(case, seed, ns)
        num = den = 0.0
        idx = _samples(ns, case["samples"], seed + 5).sum(axis=1).astype(np.float64)
        for i in range(0, len(idx), 1 << 16):
            s = idx[i:i + (1 << 16)]
            x = 1.0 / (1.0 + s)
            num += float(np.sum((x - np.exp(-np.outer(s, t)) @ w) ** 2))
            den += float(np.sum(x * x))
        return {"err": np.array([np.sqrt(num / den)])}
    entries = _entries(case, seed, _sizes(case, seed)) if case["kind"] == "cross" else None
    if entries is None:
        # the other crosses choose pivots among residuals that tie up to rounding, so their cores
        # have no value that does not hang on the order of the roundings
        return None
    cores = np.concatenate([c.reshape(-1) for c in
                            _numpy_cross(case, seed, _sizes(case, seed), entries)])
    out = np.zeros(_room(case, case["d"], case["n"]))
    out[:cores.size] = cores
    return {"ranks": None, "cores": out}

"""Performance cases of the PC-stable skeleton engine.

Each case is one pass through the public entry points as a structure-learning
program calls them, on data that a random discrete Bayesian network generates
(random DAG of about 1.25 edges per variable, in-degree at most 4, Dirichlet
conditional tables, forward sampling): the distributions that decide how many
edges survive each depth, and so how much work a skeleton is.

Kinds:

* ``ci``       explicit tests, ``fbn_ci_test`` (a program that drives its own
               constraint-based search asks for one test at a time);
* ``table``    ``fbn_ci_table``, the exact contingency table of one test;
* ``noalloc``  ``fbn_ci_test_noalloc`` on caller-owned device buffers;
* ``pairs``    ``fbn_pairwise_counts``, every pair's table at once;
* ``skeleton`` ``fbn_learn_skeleton`` and ``fbn_export_sepsets`` on data the
               handle holds;
* ``batch``    ``fbn_learn_skeleton_batch`` over many independent problems;
* ``stream``   new samples from pinned host memory into kept handles
               (``fbn_update_data_batch``), the batch of skeletons, and every
               handle's separating sets.
"""
import math

import numpy as np
import torch

import paper_2212_04259_gb300 as fbn

MAX_PARENTS = 4


# --------------------------------------------------------------------------
# inputs

def _arities(n, arity_lo, arity_hi):
    """uint8 [n], fixed by the case: what a data set of these variables has."""
    return np.random.default_rng(n * 97 + arity_hi).integers(arity_lo, arity_hi + 1, size=n).astype(np.uint8)


def _network(rng, n):
    """A random DAG in topological order 0..n-1 under a random relabelling:
    (parents per position, position -> variable)."""
    parents = [[] for _ in range(n)]
    want, have = int(round(1.25 * n)), 0
    while have < want:
        for a, b in rng.integers(0, n, size=(2 * want, 2)).tolist():
            if a == b or have >= want:
                continue
            a, b = min(a, b), max(a, b)
            if a in parents[b] or len(parents[b]) >= MAX_PARENTS:
                continue
            parents[b].append(a)
            have += 1
    return parents, rng.permutation(n)


def _samples(seed, n, n_samples, arity_lo, arity_hi, dirichlet):
    """(uint8 [n][n_samples] on the GPU, uint8 [n] arities on the host)."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)
    arities = _arities(n, arity_lo, arity_hi)
    parents, perm = _network(rng, n)
    ar = arities[perm].astype(np.int64)   # by position
    rows = max(int(np.prod([ar[p] for p in pa])) if pa else 1 for pa in parents)
    rmax = int(ar.max())
    # Dirichlet rows from unit-scale gamma draws of shape 1 or 1/2
    if dirichlet == 1.0:
        g = -torch.log(torch.rand((n, rows, rmax), device="cuda", generator=gen).clamp_min(1e-30))
    else:
        g = torch.randn((n, rows, rmax), device="cuda", generator=gen).square().mul_(0.5).clamp_min(1e-30)
    live = torch.arange(rmax, device="cuda")[None, :] < torch.as_tensor(ar, device="cuda")[:, None]
    g = g * live[:, None, :]
    cum = (g.cumsum(2) / g.sum(2, keepdim=True))[:, :, : rmax - 1].reshape(-1, rmax - 1)
    # a padded value's threshold is never passed
    dead = (torch.arange(1, rmax, device="cuda")[None, :] >= torch.as_tensor(ar, device="cuda")[:, None])
    cum = torch.where(dead[:, None, :].expand(n, rows, rmax - 1).reshape(-1, rmax - 1), torch.full_like(cum, 2.0), cum)
    level = np.zeros(n, dtype=np.int64)
    for b in range(n):
        if parents[b]:
            level[b] = 1 + max(level[p] for p in parents[b])
    data = torch.zeros((n + 1, n_samples), dtype=torch.uint8, device="cuda")   # row n: the absent parent
    for lv in range(int(level.max()) + 1):
        vs = np.nonzero(level == lv)[0]
        pa = np.full((len(vs), MAX_PARENTS), n, dtype=np.int64)
        stride = np.zeros((len(vs), MAX_PARENTS), dtype=np.int64)
        for i, v in enumerate(vs):
            s = 1
            for k, p in enumerate(parents[v]):
                pa[i, k], stride[i, k] = p, s
                s *= int(ar[p])
        pa_d, st_d = torch.as_tensor(pa, device="cuda"), torch.as_tensor(stride, device="cuda")
        vs_d = torch.as_tensor(vs, device="cuda")
        step = max(1, 40_000_000 // n_samples)
        for i in range(0, len(vs), step):   # bounded temporaries
            j = min(i + step, len(vs))
            row = (vs_d[i:j] * rows)[:, None].expand(j - i, n_samples).to(torch.int32)
            for k in range(min(MAX_PARENTS, lv * MAX_PARENTS)):
                row = row + data[pa_d[i:j, k]].to(torch.int32) * st_d[i:j, k].to(torch.int32)[:, None]
            u = torch.rand((j - i, n_samples), device="cuda", generator=gen)
            val = torch.zeros((j - i, n_samples), dtype=torch.uint8, device="cuda")
            for t in range(rmax - 1):
                val += (u >= cum[:, t][row])
            data[vs_d[i:j]] = val
    out = torch.empty((n, n_samples), dtype=torch.uint8, device="cuda")
    perm_d = torch.as_tensor(perm, device="cuda")
    out[perm_d] = data[:n]
    return out, arities


def _sep_buffers(ns):
    """Arrays for the separating sets of problems of ns variables each, one
    section per problem: pairs, offsets, members, and where each begins."""
    caps = [n * (n - 1) // 2 for n in ns]
    mem = [c * (8 if n <= 200 else 2) for n, c in zip(ns, caps)]
    at = [(sum(caps[:p]), sum(caps[:p]) + p, sum(mem[:p])) for p in range(len(ns))]
    return {"pairs": np.zeros((sum(caps), 2), np.int32), "offsets": np.zeros(sum(caps) + len(ns), np.int64),
            "members": np.zeros(sum(mem), np.int32)}, at


def _keep_seps(buf, at, h):
    """The handle's separating sets into the program's own arrays."""
    pairs, offsets, members = fbn.fbn_export_sepsets(h, as_dict=False)
    p, o, m = at
    buf["pairs"][p:p + len(pairs)] = pairs
    buf["offsets"][o:o + len(offsets)] = offsets
    buf["members"][m:m + len(members)] = members


def _problem_sizes(case):
    """(n, N) of each problem of a batch: fixed by the case, not by the seed."""
    rng = np.random.default_rng(case["sizes"])
    out = []
    for _ in range(case["problems"]):
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        N = int(round(math.exp(rng.uniform(math.log(case["N_lo"]), math.log(case["N_hi"])))))
        out.append((n, N))
    return out


def _tests(case):
    """(x, y, z) of each explicit test, fixed by the case: distinct variables;
    conditioning sets of the case's size, or cycling through 0 .. that size."""
    rng = np.random.default_rng(case["n"] * 31 + case["d"])
    out = []
    for t in range(case["tests"]):
        d = t % (case["d"] + 1) if case["spread"] else case["d"]
        vs = rng.choice(case["n"], size=d + 2, replace=False).tolist()
        out.append((vs[0], vs[1], sorted(vs[2:])))
    return out


# --------------------------------------------------------------------------
# cases

def _ci(kind, n, N, arity_hi, d, tests, spread):
    return {"kind": kind, "n": n, "N": N, "arity_lo": 2, "arity_hi": arity_hi, "dirichlet": 1.0, "d": d,
            "tests": tests, "spread": spread}


def _skel(n, N, arity_hi, dirichlet, alpha, max_depth, statistic="g2", df="fixed"):
    # the marginal graph (max_depth 0) has empty separating sets only: not read
    return {"kind": "skeleton", "n": n, "N": N, "arity_lo": 2, "arity_hi": arity_hi, "dirichlet": dirichlet,
            "alpha": alpha, "max_depth": max_depth, "statistic": statistic, "df": df, "seps": max_depth != 0}


def _batch(kind, problems, sizes, n_lo, n_hi, N_lo, N_hi):
    return {"kind": kind, "problems": problems, "sizes": sizes, "n_lo": n_lo, "n_hi": n_hi, "N_lo": N_lo,
            "N_hi": N_hi, "arity_lo": 2, "arity_hi": 4, "dirichlet": 1.0, "alpha": 0.05}


def listed():
    return [
        # one test of a search that asks for them one by one, on a small data set: call latency
        dict(_ci("ci", 20, 5000, 4, 1, 1, False), name="ci_small"),
        # a scan of tests with 0..3 conditioning variables on a large, ragged sample
        dict(_ci("ci", 40, 100003, 5, 3, 8, True), name="ci_scan"),
        # the table of one test with four conditioning variables over 200,000 samples
        dict(_ci("table", 40, 200000, 5, 4, 1, False), name="table_large"),
        # tests inside a loop that owns the device memory: queued without synchronising
        dict(_ci("noalloc", 40, 50000, 4, 2, 4, False), name="noalloc_mid"),
        # every pair's counts (pairwise dependence screens, Chow-Liu style scores)
        {"name": "pairs_300", "kind": "pairs", "n": 300, "N": 20011, "arity_lo": 2, "arity_hi": 4, "dirichlet": 1.0},
        # skeletons over the range: a small network of few samples, an ordinary one, ...
        dict(_skel(20, 5000, 4, 1.0, 0.05, -1), name="skeleton_small"),
        dict(_skel(40, 50000, 4, 0.5, 0.05, -1), name="skeleton_mid"),
        # ... Pearson's statistic with the observed table's degrees of freedom on an odd sample count, ...
        dict(_skel(101, 9973, 4, 1.0, 0.05, -1, "x2", "adjusted"), name="skeleton_x2_adjusted"),
        # ... a thousand variables to depth 4, ...
        dict(_skel(1000, 100000, 5, 0.5, 0.01, 4), name="skeleton_large"),
        # ... and the marginal tests alone of a thousand variables on 200,000 samples
        dict(_skel(1000, 200000, 5, 1.0, 0.05, 0), name="skeleton_depth0"),
        # many independent problems in one call (bootstrap replicates, one network per group)
        dict(_batch("batch", 256, 11, 20, 300, 1000, 50000), name="batch_256"),
        # fresh samples for kept handles from host memory, end to end
        dict(_batch("stream", 20, 12, 20, 300, 1000, 50000), name="stream_20"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ci", "table", "noalloc", "pairs", "skeleton", "skeleton", "skeleton", "batch", "stream"])
    if kind in ("ci", "table", "noalloc"):
        d = rng.randint(0, 5)
        return _ci(kind, rng.randint(max(8, d + 2), 64), _log_int(rng, 300, 300000), rng.randint(2, 6), d,
                   1 if kind == "table" else rng.randint(1, 8), kind != "table" and rng.random() < 0.5)
    if kind == "pairs":
        return {"kind": "pairs", "n": _log_int(rng, 10, 800), "N": _log_int(rng, 1000, 100000), "arity_lo": 2,
                "arity_hi": rng.randint(2, 6), "dirichlet": 1.0}
    if kind == "skeleton":
        stat, df = rng.choice([("g2", "fixed")] * 3 + [("x2", "fixed"), ("g2", "adjusted"), ("x2", "adjusted")])
        dirichlet = rng.choice([0.5, 1.0])
        if rng.random() < 0.25:   # many variables, stricter level, bounded depth
            return _skel(_log_int(rng, 300, 900), _log_int(rng, 5000, 90000), rng.randint(3, 5), dirichlet, 0.01,
                         rng.randint(0, 4), stat, df)
        return _skel(_log_int(rng, 10, 250), _log_int(rng, 500, 60000), rng.randint(2, 6), dirichlet,
                     rng.choice([0.01, 0.05]), rng.choice([-1, -1, 2, 3]), stat, df)
    problems = rng.randint(2, 60) if kind == "batch" else rng.randint(1, 20)
    n_lo, N_lo = rng.randint(10, 40), _log_int(rng, 500, 4000)
    return _batch(kind, problems, rng.randint(0, 10 ** 6), n_lo, rng.randint(n_lo + 10, 250), N_lo,
                  _log_int(rng, 5000, 50000))


# --------------------------------------------------------------------------
# passes

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "stream"):
        problems = [_samples(seed * 1009 + p, n, N, case["arity_lo"], case["arity_hi"], case["dirichlet"])
                    for p, (n, N) in enumerate(_problem_sizes(case))]
        handles = [fbn.fbn_create(x, a) for x, a in problems]
        sizes = [h.n * h.n for h in handles]
        # every problem's adjacency in one buffer (rows of one result array), on the device for a
        # program that goes on there, pinned for one that reads it
        host = kind == "stream"
        adj = torch.zeros(sum(sizes), dtype=torch.uint8, device="cpu" if host else "cuda", pin_memory=host)
        views, o = [], 0
        for h, s in zip(handles, sizes):
            views.append(adj[o:o + s].view(h.n, h.n))
            o += s
        fresh = [x.cpu().pin_memory() for x, _ in problems] if host else None
        buf, at = _sep_buffers([h.n for h in handles]) if host else (None, None)
        return {"case": case, "handles": handles, "adj": adj, "views": views, "fresh": fresh, "seps": buf, "at": at}
    data, arities = _samples(seed, case["n"], case["N"], case["arity_lo"], case["arity_hi"], case["dirichlet"])
    s = {"case": case}
    if kind in ("ci", "table", "noalloc"):
        s["tests"] = _tests(case)
    if kind == "noalloc":
        ld = (case["N"] + 15) // 16 * 16
        s["data"] = torch.zeros((case["n"], ld), dtype=torch.uint8, device="cuda")
        s["data"][:, : case["N"]] = data
        s["ld"], s["arities"] = ld, arities
        s["out"] = torch.zeros((case["tests"], 3), dtype=torch.float64, device="cuda")
        return s
    if kind == "skeleton":
        s["h"] = fbn.fbn_create(data, arities, statistic=case["statistic"], df=case["df"])
        s["adj"] = torch.zeros((case["n"], case["n"]), dtype=torch.uint8).pin_memory()
        if case["seps"]:
            s["seps"], s["at"] = _sep_buffers([case["n"]])
    else:
        s["h"] = fbn.fbn_create(data, arities)
    if kind == "pairs":
        M = int(arities.astype(np.int64).sum())
        s["counts"] = torch.zeros((M, M), dtype=torch.int32, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "ci":
        r = np.array([fbn.fbn_ci_test(s["h"], x, y, z) for x, y, z in s["tests"]])
        return {"g2": r[:, 0], "df": r[:, 1], "p": r[:, 2]}
    if kind == "table":
        return [fbn.fbn_ci_table(s["h"], x, y, z) for x, y, z in s["tests"]]
    if kind == "noalloc":
        for t, (x, y, z) in enumerate(s["tests"]):
            fbn.fbn_ci_test_noalloc(s["data"], s["ld"], case["N"], s["arities"], x, y, z, s["out"][t])
        return {"g2": s["out"][:, 0], "df": s["out"][:, 1], "p": s["out"][:, 2]}
    if kind == "pairs":
        return fbn.fbn_pairwise_counts(s["h"], s["counts"])
    if kind == "skeleton":
        adj = fbn.fbn_learn_skeleton(s["h"], case["alpha"], case["max_depth"], s["adj"])
        if not case["seps"]:
            return adj
        _keep_seps(s["seps"], s["at"][0], s["h"])
        return {"adj": adj, **s["seps"]}
    if kind == "stream":
        fbn.fbn_update_data_batch(s["handles"], s["fresh"])
    fbn.fbn_learn_skeleton_batch(s["handles"], case["alpha"], -1, s["views"])
    if kind == "batch":
        return s["adj"]
    for h, at in zip(s["handles"], s["at"]):
        _keep_seps(s["seps"], at, h)
    return {"adj": s["adj"], **s["seps"]}


# --------------------------------------------------------------------------
# what a pass cannot do without

def work(case):
    """Bytes: every sample read once and the results written once.  Operations:
    one count per sample and test; of a skeleton, those of depth 0 (every
    pair), since the later depths depend on the data."""
    kind = case["kind"]
    if kind in ("ci", "table", "noalloc"):
        mean = 0.5 * (case["arity_lo"] + case["arity_hi"])
        rows = sum((t % (case["d"] + 1) if case["spread"] else case["d"]) + 2 for t in range(case["tests"]))
        out = 4.0 * mean ** (case["d"] + 2) if kind == "table" else 24.0 * case["tests"]
        return {"bytes": rows * case["N"] + out, "flops": case["tests"] * case["N"]}
    if kind == "pairs":
        m = case["n"] * 0.5 * (case["arity_lo"] + case["arity_hi"])
        return {"bytes": case["n"] * case["N"] + 4.0 * m * m, "flops": case["n"] * (case["n"] - 1) / 2 * case["N"]}
    sizes = [(case["n"], case["N"])] if kind == "skeleton" else _problem_sizes(case)
    return {"bytes": sum(n * N + n * n for n, N in sizes), "flops": sum(n * (n - 1) / 2 * N for n, N in sizes)}


def tolerance(case):
    """Counts, graphs and separating sets are whole numbers.  The statistic and
    its p-value are 64-bit: sums in another order move them by about 1e-14
    (the p-value by that times its condition, the statistic's size)."""
    return {"rel": 1e-10} if case["kind"] in ("ci", "noalloc") else "exact"


def exact(case, seed):
    """G^2, degrees of freedom and p in 64 bits for the explicit tests, from
    plain counts; tables and pair counts likewise.  The skeletons are whole
    numbers, compared between implementations as they are."""
    kind = case["kind"]
    if kind not in ("ci", "table", "noalloc", "pairs"):
        return None
    data, arities = _samples(seed, case["n"], case["N"], case["arity_lo"], case["arity_hi"], case["dirichlet"])
    if kind == "pairs":
        onehot = torch.cat([(data[v][None, :] == torch.arange(int(a), device="cuda")[:, None])
                            for v, a in enumerate(arities)]).double()
        return (onehot @ onehot.T).round().to(torch.int32)
    out = []
    for x, y, z in _tests(case):
        rows = [*z, x, y]
        idx = torch.zeros(case["N"], dtype=torch.int64, device="cuda")
        for v in rows:
            idx = idx * int(arities[v]) + data[v].to(torch.int64)
        rx, ry = int(arities[x]), int(arities[y])
        nz = int(np.prod([int(arities[v]) for v in z], dtype=np.int64)) if z else 1
        counts = torch.bincount(idx, minlength=nz * rx * ry)
        if kind == "table":
            out.append(counts.to(torch.int32))
            continue
        t = counts.cpu().double().view(nz, rx, ry)
        nx, ny, nn = t.sum(2, keepdim=True), t.sum(1, keepdim=True), t.sum((1, 2), keepdim=True)
        e = nx * ny
        # the log of the ratio as log1p of the exact difference over the denominator
        lr = torch.log1p(torch.where(t > 0, (t * nn - e) / e.clamp_min(1.0), torch.zeros_like(t)))
        g2 = 2.0 * float((t * lr).sum())
        df = float((rx - 1) * (ry - 1) * nz)
        p = float(torch.special.gammaincc(torch.tensor(df / 2, dtype=torch.float64),
                                          torch.tensor(max(g2, 0.0) / 2, dtype=torch.float64)))
        out.append((g2, df, p))
    if kind == "table":
        return out
    r = np.array(out)
    return {"g2": r[:, 0], "df": r[:, 1], "p": r[:, 2]}

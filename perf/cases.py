"""The work a user has this library do, as cases that can be timed.

Every case is one call sequence of the public Python binding on a synthetic graph of the
families the repository's own benchmark, tests and workload definitions use (Erdos-Renyi,
Chung-Lu power law, stochastic block model, R-MAT, batches of uneven power-law graphs).
The graphs are drawn here on the GPU from the seed alone, with the same recipes as the
host generators (which take many seconds at these sizes).

    listed()             the cases
    draw(rng)            another case of the same ranges
    prepare(case, seed)  what a program holds before the call (inputs or resident handle)
    run(state)           one pass
    work(case)           bytes and operations a pass cannot do without
    exact(case, seed)    None: every output is a whole number (or that number scaled by an
                         exact power of the colours), compared digit by digit
"""
import math

import numpy as np
import torch

import paper_1403_0734_gb300 as kc

DEV = "cuda"


def listed():
    return [
        # One small graph handed over as host arrays, triangles wanted: the smallest whole
        # call (copy in, orientation, count, answer), where launches and waits are all there is.
        {"name": "er_1k_oneshot_k3", "op": "one_shot", "graph": "er", "n": 1000, "m": 10000, "k": 3},
        # A small resident graph asked for one number, as a server does all day.
        {"name": "chunglu_20k_k4", "op": "count", "graph": "chung_lu", "n": 20000, "m": 200000, "k": 4,
         "wmax": 2000.0, "outputs": False},
        # A large power-law graph that arrives on the device and is read once: orientation
        # and triangles with the per-vertex and per-owner arrays.
        {"name": "chunglu_1m_orient_k3", "op": "orient_count", "graph": "chung_lu", "n": 1000000, "m": 20000000,
         "k": 3, "wmax": 20000.0, "outputs": True},
        # The same graph resident, exact counts at growing k: 4 is bound by building the
        # neighbourhoods, 5 is between, 6 by the search inside the dense hub cores.
        {"name": "chunglu_1m_k4_arrays", "op": "count", "graph": "chung_lu", "n": 1000000, "m": 20000000, "k": 4,
         "wmax": 20000.0, "outputs": True},
        {"name": "chunglu_1m_k5", "op": "count", "graph": "chung_lu", "n": 1000000, "m": 20000000, "k": 5,
         "wmax": 20000.0, "outputs": False},
        {"name": "chunglu_1m_k6_arrays", "op": "count", "graph": "chung_lu", "n": 1000000, "m": 20000000, "k": 6,
         "wmax": 20000.0, "outputs": True},
        # The colour-sampling estimate on the same graph, for when the exact count is too dear.
        {"name": "chunglu_1m_estimate_c8_k6", "op": "estimate", "graph": "chung_lu", "n": 1000000, "m": 20000000,
         "k": 6, "wmax": 20000.0, "colours": 8},
        # Community graph: no hubs, millions of small neighbourhoods, an adjacency that does
        # not fit the L2 cache.
        {"name": "sbm_2m_k5", "op": "count", "graph": "sbm", "n": 2000000, "m": 50000000, "k": 5, "p_in": 0.3,
         "outputs": False},
        # Fully dense communities, large k, with the plan the library's tuner measured once.
        {"name": "sbm_2m_dense_k7_tuned", "op": "count", "graph": "sbm", "n": 2000000, "m": 50000000, "k": 7,
         "p_in": 1.0, "outputs": True, "tuned": True},
        # R-MAT graph of the serving workload at its largest, wide hubs at an ordinary k.
        {"name": "rmat_s20_k4", "op": "count", "graph": "rmat", "scale": 20, "factor": 16, "k": 4, "outputs": False},
        # Thousands of uneven graphs counted together.
        {"name": "batch_8192_k4", "op": "batch", "graph": "batch", "graphs": 8192, "nmin": 50, "nmax": 20000, "k": 4},
        # Every clique itself, kept on the device by the program that asked for them.
        {"name": "chunglu_20k_list_k4", "op": "list", "graph": "chung_lu", "n": 20000, "m": 200000, "k": 4,
         "wmax": 2000.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["one_shot", "count", "count", "orient_count", "estimate", "sbm", "rmat", "batch", "list"])
    if op == "one_shot":
        n = _log(rng, 100, 20000)
        return {"op": op, "graph": "er", "n": n, "m": min(int(n * rng.uniform(4, 32)), n * (n - 1) // 4), "k": 3}
    if op == "sbm":
        n = 50 * _log(rng, 400, 38000)
        tuned = rng.random() < 0.3
        return {"op": "count", "graph": "sbm", "n": n, "m": 25 * n, "k": rng.randint(4, 7 if tuned else 6),
                "p_in": 1.0 if tuned else rng.choice([0.3, 0.5]), "outputs": tuned or rng.random() < 0.5, "tuned": tuned}
    if op == "rmat":
        return {"op": rng.choice(["count", "orient_count"]), "graph": "rmat", "scale": rng.randint(10, 19),
                "factor": rng.randint(8, 16), "k": rng.randint(3, 4), "outputs": True}
    if op == "batch":
        return {"op": op, "graph": "batch", "graphs": _log(rng, 60, 4000), "nmin": 50, "nmax": _log(rng, 500, 20000), "k": rng.randint(3, 5)}
    if op == "list":
        n = _log(rng, 1000, 20000)
        return {"op": op, "graph": "chung_lu", "n": n, "m": 10 * n, "k": rng.randint(3, 4), "wmax": 0.1 * n}
    n = _log(rng, 5000, 900000)
    case = {"op": op, "graph": "chung_lu", "n": n, "m": int(n * rng.uniform(8, 20)), "wmax": 0.02 * n if n > 100000 else 0.1 * n}
    if op == "estimate":
        return {**case, "k": rng.randint(4, 6), "colours": rng.randint(4, 16)}
    return {**case, "k": rng.randint(3, 4) if op == "orient_count" else rng.randint(3, 6), "outputs": rng.random() < 0.6}


# ---------------------------------------------------------------- graphs

def _csr(n, u, v):
    """Canonical CSR (symmetric, simple, sorted rows) of the pairs u, v on the GPU."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v))
    lo, hi = key // n, key % n
    key = torch.sort(torch.cat([lo * n + hi, hi * n + lo])).values
    off = torch.searchsorted(key, torch.arange(n + 1, device=DEV, dtype=torch.int64) * n)
    return off, (key % n).to(torch.int32)


def _power_offset(n, m, gamma, wmax):
    """i0 of the weights (i + i0)^(-1/(gamma-1)), i < n, whose largest is wmax when they sum to 2m."""
    s = 1.0 / (gamma - 1.0)
    want = wmax / (2.0 * m)
    lo, hi = np.full_like(want, 1e-6), n.astype(np.float64)
    for _ in range(80):
        mid = np.sqrt(lo * hi)
        share = mid ** -s * (1 - s) / ((n + mid) ** (1 - s) - mid ** (1 - s))
        lo, hi = np.where(share > want, mid, lo), np.where(share > want, hi, mid)
    return lo


def _power_ends(gen, n, i0, gamma, num):
    """num endpoints with density (x + i0)^(-s) on [0, n): n, i0 scalars or one value for each endpoint."""
    t = 1.0 - 1.0 / (gamma - 1.0)
    a = i0 ** t
    b = (n + i0) ** t
    x = (a + torch.rand(num, device=DEV, dtype=torch.float64, generator=gen) * (b - a)) ** (1.0 / t) - i0
    return torch.minimum(x.clamp_(min=0).to(torch.int64), torch.as_tensor(n - 1, device=DEV).to(torch.int64))


def _chung_lu(gen, n, m, gamma, wmax):
    i0 = float(_power_offset(np.array([n]), np.array([m]), gamma, np.array([wmax]))[0])
    ids = torch.randperm(n, device=DEV, generator=gen)
    return _csr(n, ids[_power_ends(gen, n, i0, gamma, m)], ids[_power_ends(gen, n, i0, gamma, m)])


def _er(gen, n, m):
    u = torch.randint(n, (m + m // 8 + 16,), device=DEV, generator=gen)
    v = torch.randint(n, (m + m // 8 + 16,), device=DEV, generator=gen)
    keep = u != v
    key = torch.unique(torch.minimum(u, v)[keep] * n + torch.maximum(u, v)[keep])
    key = key[torch.randperm(key.numel(), device=DEV, generator=gen)[:m]]
    return _csr(n, key // n, key % n)


def _sbm(gen, n, m, p_in, block=50):
    iu = torch.triu_indices(block, block, 1, device=DEV)
    nb = n // block
    at = torch.nonzero(torch.rand(nb, iu.shape[1], device=DEV, generator=gen) < p_in)
    u, v = iu[0][at[:, 1]] + at[:, 0] * block, iu[1][at[:, 1]] + at[:, 0] * block
    more = max(0, m - u.numel())
    x, y = (torch.randint(n, (more,), device=DEV, generator=gen) for _ in range(2))
    ids = torch.randperm(n, device=DEV, generator=gen)
    return _csr(n, ids[torch.cat([u, x])], ids[torch.cat([v, y])])


def _rmat(gen, scale, factor, a=0.57, b=0.19, c=0.19):
    n, num = 1 << scale, factor << scale
    u = torch.zeros(num, device=DEV, dtype=torch.int64)
    v = torch.zeros(num, device=DEV, dtype=torch.int64)
    for _ in range(scale):
        r = torch.rand(num, device=DEV, generator=gen)
        u = 2 * u + (r >= a + b)
        v = 2 * v + (((r >= a) & (r < a + b)) | (r >= a + b + c))
    ids = torch.randperm(n, device=DEV, generator=gen)
    return _csr(n, ids[u], ids[v])


def _batch_sizes(case, seed):
    rng = np.random.default_rng(seed)
    num = case["graphs"]
    n = np.rint(np.exp(rng.uniform(math.log(case["nmin"]), math.log(case["nmax"]), num))).astype(np.int64)
    m = np.minimum((n * rng.uniform(8, 64, num) / 2).astype(np.int64), n * (n - 1) // 2)
    return n, m


def _batch(case, seed, gen, gamma=2.3):
    """Resident handles of the batch's graphs: drawn together, a thousand or so at a time."""
    n, m = _batch_sizes(case, seed)
    i0 = _power_offset(n, m, gamma, np.sqrt(2.0 * m))
    graphs = []
    for g0 in range(0, len(n), 1024):
        gn, gm = n[g0:g0 + 1024], m[g0:g0 + 1024]
        base = np.concatenate([[0], np.cumsum(gn)])
        dn, db, di = (torch.from_numpy(x).to(DEV) for x in (gn, base[:-1], i0[g0:g0 + 1024]))
        which = torch.repeat_interleave(torch.arange(len(gn), device=DEV), torch.from_numpy(gm).to(DEV))
        u, v = (_power_ends(gen, dn[which], di[which], gamma, which.numel()) + db[which] for _ in range(2))
        ids = torch.randperm(int(base[-1]), device=DEV, generator=gen)  # shuffled inside each graph
        ids = torch.argsort(ids + torch.repeat_interleave(torch.arange(len(gn), device=DEV), dn) * int(base[-1]))
        off, adj = _csr(int(base[-1]), ids[u], ids[v])
        local = adj - torch.repeat_interleave(torch.repeat_interleave(db, dn).to(torch.int32), off.diff())
        ends = off[torch.from_numpy(base).to(DEV)].tolist()
        for i in range(len(gn)):
            o = off[int(base[i]):int(base[i + 1]) + 1] - ends[i]
            graphs.append(kc.orient(o, local[ends[i]:ends[i + 1]].clone()))
    torch.cuda.synchronize()
    return graphs


def _graph(case, gen):
    kind = case["graph"]
    if kind == "er":
        return _er(gen, case["n"], case["m"])
    if kind == "chung_lu":
        return _chung_lu(gen, case["n"], case["m"], 2.1, case["wmax"])
    if kind == "sbm":
        return _sbm(gen, case["n"], case["m"], case["p_in"])
    return _rmat(gen, case["scale"], case["factor"])


# ---------------------------------------------------------------- cases

def _arrays(n, wanted):
    """Output buffers a program keeps: the total's two words, and the two arrays."""
    one = lambda: torch.zeros(n, device=DEV, dtype=torch.int64)  # noqa: E731
    return torch.zeros(2, device=DEV, dtype=torch.int64), one() if wanted else None, one() if wanted else None


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    op, st = case["op"], {"op": case["op"], "k": case["k"]}
    if op == "batch":
        st["graphs"] = _batch(case, seed, gen)
        return st
    off, adj = _graph(case, gen)
    n = off.numel() - 1
    if op == "one_shot":
        st["off"], st["adj"] = off.cpu().numpy(), adj.cpu().numpy()
        return st
    if op == "orient_count":
        st["off"], st["adj"] = off, adj
        st["out"] = _arrays(n, case["outputs"])
        return st
    st["g"] = kc.orient(off, adj)
    torch.cuda.synchronize()  # the graph is resident: its input may go
    if op == "list":
        st["run"] = torch.empty((1 << 20, case["k"]), device=DEV, dtype=torch.int32)  # one run of cliques
        st["rows"] = torch.full((1 << 24, case["k"]), -1, device=DEV, dtype=torch.int32)
    if op == "estimate":
        st["colours"], st["seed"] = case["colours"], seed
    if op == "count":
        st["out"] = _arrays(n, True) if case["outputs"] else None
        if case.get("tuned"):
            kc.set_tuning(st["g"], kc.tune(st["g"], case["k"], per_vertex=case["outputs"]))
    return st


def run(st):
    op, k = st["op"], st["k"]
    if op == "one_shot":
        total, pv, po = kc.count_csr(st["off"], st["adj"], k, per_vertex=True, per_owner=True)
        return {"total": total, "per_vertex": pv.view(np.int64), "per_owner": po.view(np.int64)}
    if op == "orient_count":
        g = kc.orient(st["off"], st["adj"])
        kc.count_device(g, k, *st["out"])
        return [t for t in st["out"] if t is not None]
    if op == "count":
        if st["out"] is None:
            return kc.count(st["g"], k)[0]
        kc.count_device(st["g"], k, *st["out"])
        return list(st["out"])
    if op == "estimate":
        sampled, estimate, po = kc.estimate(st["g"], k, st["colours"], st["seed"], per_owner=True)
        return {"sampled": sampled, "estimate": estimate, "per_owner": po.view(np.int64)}
    if op == "batch":
        return np.array(kc.count_batch(st["graphs"], k), dtype=np.int64)
    at = 0

    def keep(got):
        nonlocal at
        st["rows"][at:at + got[1]].copy_(st["run"][:got[1]])
        at += got[1]

    kc.list_runs(st["g"], k, keep, cap=st["run"].shape[0], device_buffer=st["run"])
    return st["rows"]


def work(case):
    """Each row of the oriented graph read once (or of the input, where the pass orients it), each
    output written once; the operations depend on the drawn graph and are left at none."""
    if case["graph"] == "batch":
        n, m = (float(x.sum()) for x in _batch_sizes(case, 1))
        return {"bytes": 4 * m + 8 * n + 8 * case["graphs"], "flops": 0.0}
    n = float(1 << case["scale"] if case["graph"] == "rmat" else case["n"])
    m = float(case["factor"] * n if case["graph"] == "rmat" else case["m"])
    size = 4 * m + 8 * n                            # Gamma+ rows and their offsets
    if case["op"] in ("one_shot", "orient_count"):
        size += 8 * m + 8 * n                       # the input
    if case["op"] == "one_shot" or case.get("outputs"):
        size += 16 * n                              # both arrays
    if case["op"] == "estimate":
        size += 8 * n
    return {"bytes": size, "flops": 0.0}


def exact(case, seed):
    return None

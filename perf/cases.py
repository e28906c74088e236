"""Workloads of the library for timing: each case is one call sequence a user's
program makes through the package's public entry points, with the inputs it
would hold on the GPU (graphs registered once, sampled-edge lists, weights).

Graphs are made on the GPU from the seed alone with the models of the
repository's configurations (Erdos-Renyi, Chung-Lu, R-MAT, random geometric).
"""
import math
from fractions import Fraction

import numpy as np
import torch

import paper_1701_01772_gb300 as gs

GIB = 1 << 30
FOUR = tuple(1 << g for g in gs.GRAPHLETS)
D = (3, 2, 6, 1, 2, 4, 6, 1)
D_DISC = (1, 6, 6, 2, 2, 1, 12)


# ------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest configuration: exact counts of one small graph, where
        # launches and waits are the time
        dict(name="er_2k_exact", op="count", model="er", n=2000, m=20000),
        # a caller's own shuffled edge list on a small heavy-tailed graph, with
        # the disconnected graphlets and per-edge counts
        dict(name="cl_20k_explicit", op="explicit", model="cl", n=20000, m=150000, cap=1500,
             fraction=0.05),
        # the power-law configuration: a 1% estimate on a resident graph with
        # the default index
        dict(name="cl_1m_1pct", op="estimate", model="cl", n=1000000, m=20000000, cap=50000,
             fraction=0.01),
        # the same graph counted exactly, sharing the GPU (20 GiB index): the
        # largest call
        dict(name="cl_1m_exact", op="count", model="cl", n=1000000, m=20000000, cap=50000,
             budget_gib=20),
        # exact triangles and 2-stars of every edge of an R-MAT graph
        dict(name="rmat_22_exact3", op="count3", model="rmat", scale=22, edge_factor=16,
             budget_gib=20),
        # the headline graph, a 0.1% estimate, with the index it has when
        # served beside others
        dict(name="rmat_24_0p1pct", op="estimate", model="rmat", scale=24, edge_factor=16,
             fraction=0.001, budget_gib=20),
        # micro-level statistics (Algorithm 7) of a sample, a tenth of the
        # neighbours probed
        dict(name="cl_100k_micro", op="micro", model="cl", n=100000, m=2000000, cap=50000,
             fraction=0.01, p_e=0.1),
        # k-core numbers, a sample weighted by them and its Horvitz-Thompson
        # estimates
        dict(name="cl_100k_kcore", op="weighted", model="cl", n=100000, m=2000000, cap=50000,
             fraction=0.01),
        # adaptive estimation (Algorithm 8) until the estimates settle
        dict(name="rmat_18_adaptive", op="adaptive", model="rmat", scale=18, edge_factor=16,
             beta=0.02, t_max=12),
        # a batch of uneven small graphs, exact counts for each
        dict(name="batch_1024", op="batch", count=1024, n_lo=50, n_hi=5000, deg_lo=4, deg_hi=40),
        # a graph seen once: registration with its checks and index, exact
        # triangles and 2-stars, release
        dict(name="cl_100k_register", op="register", model="cl", n=100000, m=2000000, cap=50000),
        # requests of several graphs and sample sizes through the server
        dict(name="served_32", op="serve", requests=32, f_lo=0.001, f_hi=0.1, scale=14),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _graph(rng, m_lo, m_hi, n_min=300):
    """A drawn graph of about m_lo..m_hi edges."""
    m = int(_log(rng, m_lo, m_hi))
    model = rng.choice(("er", "cl", "cl", "rmat"))
    if model == "rmat":
        ef = rng.randint(6, 20)
        return dict(model="rmat", scale=max(9, int(round(math.log2(m / ef)))), edge_factor=ef)
    n = max(n_min, int(m / rng.uniform(5, 25)))
    if model == "er":
        return dict(model="er", n=n, m=min(m, n * (n - 1) // 4))
    return dict(model="cl", n=n, m=m, cap=int(n * rng.uniform(0.02, 0.15)) + 8)


def draw(rng):
    op = rng.choice(("count", "count3", "estimate", "estimate", "explicit", "micro", "weighted",
                     "adaptive", "batch", "register", "serve"))
    budget = dict(budget_gib=rng.choice((2, 5, 20)))
    if op == "batch":
        n_hi = rng.randint(300, 5000)
        return dict(op=op, count=int(_log(rng, 17, 1024)), n_lo=rng.randint(10, 200), n_hi=n_hi,
                    deg_lo=rng.randint(2, 8), deg_hi=rng.randint(12, 40))
    if op == "serve":
        return dict(op=op, requests=rng.randint(3, 32), f_lo=0.001, f_hi=rng.choice((0.03, 0.1)),
                    scale=rng.randint(11, 14))
    if op == "count":
        return dict(op=op, **_graph(rng, 3e3, 4e6), **budget)
    if op == "count3":
        return dict(op=op, **_graph(rng, 3e3, 6e7), **budget)
    if op == "register":
        return dict(op=op, **_graph(rng, 1e4, 3e6), **budget)
    g = _graph(rng, 1e4, 1e7)
    if op == "adaptive":
        return dict(op=op, **g, **budget, beta=rng.choice((0.01, 0.05)), t_max=rng.randint(4, 12))
    if op == "micro":
        return dict(op=op, **_graph(rng, 1e4, 2e6), **budget, fraction=_log(rng, 0.001, 0.01),
                    p_e=rng.choice((0.02, 0.1, 0.3, 1.0)))
    if op == "weighted":
        return dict(op=op, **_graph(rng, 1e4, 4e6), **budget, fraction=_log(rng, 0.001, 0.03))
    return dict(op=op, **g, **budget, fraction=_log(rng, 0.001, 0.1))


# ------------------------------------------------------------------- graphs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & (2**62 - 1))
    return g


def _rand(k, g):
    return torch.rand(k, generator=g, device="cuda", dtype=torch.float64)


def _unique(keys):
    keys = torch.sort(keys).values
    if keys.numel() == 0:
        return keys
    keep = torch.ones_like(keys, dtype=torch.bool)
    torch.ne(keys[1:], keys[:-1], out=keep[1:])
    return keys[keep]


def _pair_keys(a, b, n):
    """Sorted distinct keys min * n + max of the pairs that are no loops."""
    lo, hi = torch.minimum(a, b), torch.maximum(a, b)
    return _unique((lo * n + hi)[lo != hi])


def _csr(keys, n):
    """CSR (int64 row offsets, int32 sorted adjacency) of distinct pair keys."""
    lo, hi = keys // n, keys % n
    both = torch.sort(torch.cat((keys, hi * n + lo))).values
    row = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row[1:] = torch.cumsum(torch.bincount(both // n, minlength=n), 0)
    return row, (both % n).to(torch.int32)


def _cl_weights(n, m, gamma, cap):
    """Capped power-law weights c (i + 1)^(-1 / (gamma - 1)) summing to 2m."""
    w = torch.arange(1, n + 1, device="cuda", dtype=torch.float64) ** (-1.0 / (gamma - 1.0))
    cap, c = min(float(cap), n / 2.0), 2.0 * m / float(w.sum())
    for _ in range(30):
        c *= 2.0 * m / float(torch.clamp(c * w, max=cap).sum())
    return torch.clamp(c * w, max=cap)


def _edges(case, g):
    """Distinct pair keys and the vertex count of a case's graph."""
    if case["model"] == "rmat":
        scale = case["scale"]
        n, k = 1 << scale, case["edge_factor"] << scale
        a = torch.zeros(k, dtype=torch.int64, device="cuda")
        b = torch.zeros(k, dtype=torch.int64, device="cuda")
        for _ in range(scale):
            r = torch.rand(k, generator=g, device="cuda")
            low = r >= 0.76
            a.mul_(2).add_(low)
            b.mul_(2).add_(((r >= 0.57) & ~low) | (r >= 0.95))
            del r, low
        perm = torch.randperm(n, generator=g, device="cuda")
        return _pair_keys(perm[a], perm[b], n), n
    n, m = case["n"], case["m"]
    perm = torch.randperm(n, generator=g, device="cuda")
    cum = None
    if case["model"] == "cl":
        cum = torch.cumsum(_cl_weights(n, m, 2.1, case["cap"]), 0)

    def ends(k):
        if cum is None:
            return torch.randint(n, (k,), generator=g, device="cuda")
        return perm[torch.searchsorted(cum, _rand(k, g) * cum[-1]).clamp_(max=n - 1)]

    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    k = m
    for _ in range(6):
        keys = _unique(torch.cat((keys, _pair_keys(ends(k), ends(k), n))))
        if keys.numel() >= 0.999 * m:
            break
        k = int((m - keys.numel()) * 1.5) + 16
    if keys.numel() > m:
        keys = keys[torch.sort(torch.randperm(keys.numel(), generator=g, device="cuda")[:m]).values]
    return keys, n


def _expand(start, count):
    """For each i the positions start[i] .. start[i] + count[i] - 1: (i, position)."""
    i = torch.repeat_interleave(torch.arange(count.numel(), device="cuda"), count)
    first = torch.cumsum(count, 0) - count
    return i, torch.arange(i.numel(), device="cuda") - first[i] + start[i]


def _batch_graphs(case, seed):
    """Packed CSR of small Erdos-Renyi, Chung-Lu 2.3 and geometric graphs."""
    rng = np.random.RandomState(int(seed) & 0x7FFFFFFF)
    G = case["count"]
    kind = rng.randint(0, 3, G)
    ns = rng.randint(case["n_lo"], case["n_hi"] + 1, G).astype(np.int64)
    deg = np.minimum(rng.uniform(case["deg_lo"], case["deg_hi"], G), (ns - 1) / 2.0)
    g = _gen(seed)
    dev = lambda x: torch.as_tensor(x, device="cuda")  # noqa: E731
    off = np.concatenate(([0], np.cumsum(ns)))
    N = int(off[-1])
    n_t, off_t, kind_t = dev(ns), dev(off), dev(kind)
    gid = torch.repeat_interleave(torch.arange(G, device="cuda"), n_t)
    loc = torch.arange(N, device="cuda") - off_t[gid]
    # Erdos-Renyi and Chung-Lu: endpoints drawn by vertex weight in each graph
    w = torch.where(kind_t[gid] == 1, (loc + 1).double() ** (-1.0 / 1.3), torch.ones_like(loc).double())
    tot = torch.zeros(G, dtype=torch.float64, device="cuda").index_add_(0, gid, w)
    cap = n_t.double() / 2 / (n_t.double() * dev(deg))  # of the graph's weight
    w = torch.minimum(w / tot[gid], cap[gid])
    cum = torch.cumsum(w, 0)
    cum0 = torch.cat((torch.zeros(1, dtype=torch.float64, device="cuda"), cum))
    draws = dev(np.where(kind == 2, 0, np.round(ns * deg / 2)).astype(np.int64))
    eg = torch.repeat_interleave(torch.arange(G, device="cuda"), draws)
    lo_c, hi_c = cum0[off_t[eg]], cum0[off_t[eg + 1]]

    def ends():
        x = torch.searchsorted(cum, lo_c + (hi_c - lo_c) * _rand(eg.numel(), g), right=True)
        return torch.minimum(torch.maximum(x, off_t[eg]), off_t[eg + 1] - 1)

    a, b = ends(), ends()
    # geometric graphs: candidates from the 3 x 3 cells around each point
    p = torch.nonzero(kind_t[gid] == 2).squeeze(1)
    pg = gid[p]
    r = torch.sqrt(dev(deg) / (math.pi * n_t.double()))
    gc = torch.clamp((1.0 / r).long(), min=1, max=64)
    x, y = _rand(p.numel(), g), _rand(p.numel(), g)
    cx = torch.minimum((x * gc[pg]).long(), gc[pg] - 1)
    cy = torch.minimum((y * gc[pg]).long(), gc[pg] - 1)
    coff = torch.cumsum(gc * gc, 0) - gc * gc
    cell = coff[pg] + cy * gc[pg] + cx
    order = torch.argsort(cell, stable=True)
    p, pg, x, y, cx, cy, cell = (v[order] for v in (p, pg, x, y, cx, cy, cell))
    cells = int((gc * gc).sum())
    cs = torch.zeros(cells + 1, dtype=torch.int64, device="cuda")
    cs[1:] = torch.cumsum(torch.bincount(cell, minlength=cells), 0)
    pa, pb = [a], [b]
    for dy in (-1, 0, 1):
        row = cy + dy
        ok = (row >= 0) & (row < gc[pg])
        base = coff[pg] + torch.clamp(row, min=0) * gc[pg]
        base = torch.where(ok, base, coff[pg])
        s = cs[base + torch.clamp(cx - 1, min=0)]
        e = cs[base + torch.minimum(cx + 1, gc[pg] - 1) + 1]
        i, j = _expand(s, torch.where(ok, e - s, torch.zeros_like(s)))
        near = (i < j) & ((x[i] - x[j]) ** 2 + (y[i] - y[j]) ** 2 < r[pg[i]] ** 2)
        pa.append(p[i[near]])
        pb.append(p[j[near]])
    # labels permuted inside each graph
    shuffled = torch.argsort(gid.double() + 0.999 * _rand(N, g))
    keys = _pair_keys(shuffled[torch.cat(pa)], shuffled[torch.cat(pb)], N)
    row, col = _csr(keys, N)
    owner = torch.repeat_interleave(gid, row[1:] - row[:-1])
    return off_t, row, (col - off_t[owner]).to(torch.int32)


def _upper(row, col):
    """Canonical edges (u < v) in row-major order, int32 [M, 2]."""
    n = row.numel() - 1
    src = torch.repeat_interleave(torch.arange(n, device="cuda", dtype=torch.int32), row[1:] - row[:-1])
    keep = src < col
    return torch.stack((src[keep], col[keep]), 1)


def _sample(case, seed, row, col):
    """A shuffled edge list with random orientations: a fixed share of the
    edges asked for."""
    g = _gen(seed + 1)
    up = _upper(row, col)
    up = up[torch.randperm(up.shape[0], generator=g, device="cuda")[:int(_size(case)[1] * case["fraction"])]]
    return torch.where((_rand(up.shape[0], g) < 0.5)[:, None], up.flip(1), up).contiguous()


# ------------------------------------------------------------------- state

def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        off, row, col = _batch_graphs(case, seed)
        torch.cuda.empty_cache()
        return dict(case=case, batch=gs.Batch(off, row, col, autotune=False))
    if op == "serve":
        graphs = [dict(model="er", n=2000, m=20000),
                  dict(model="cl", n=20000, m=150000, cap=1500),
                  dict(model="rmat", scale=case["scale"], edge_factor=12),
                  dict(model="cl", n=100000, m=2000000, cap=50000)]
        srv = gs.Server(hbm_budget_bytes=40 * GIB, max_batch=64, lanes=2)
        for k, c in enumerate(graphs):
            srv.add_graph(*_csr(*_edges(c, _gen(seed * 16 + k))))
        torch.cuda.empty_cache()
        srv.start(hub_budget_bytes=5 * GIB)
        rng = np.random.RandomState(int(seed) & 0x7FFFFFFF)
        reqs = []
        for k in range(case["requests"]):
            f = math.exp(rng.uniform(math.log(case["f_lo"]), math.log(case["f_hi"])))
            mask = gs.GS_THREE_NODE if rng.rand() < 0.3 else gs.GS_CONNECTED
            reqs.append((int(rng.randint(4)), f, int(rng.randint(1 << 31)), mask))
        return dict(case=case, server=srv, requests=reqs)
    row, col = _csr(*_edges(case, _gen(seed)))
    budget = int(case.get("budget_gib", 0)) * GIB
    state = dict(case=case, seed=int(seed) & (2**63 - 1), row=row, col=col, budget=budget)
    if op == "explicit" or op == "micro":
        keep = state["pairs"] = _sample(case, seed, row, col)
        if op == "micro":
            state["x"] = torch.empty((keep.shape[0], 15), dtype=torch.float64, device="cuda")
    torch.cuda.empty_cache()
    if op != "register":
        state["graph"] = gs.Graph(row, col, hub_budget_bytes=budget)
    if op == "weighted":
        G = state["graph"]
        state["core"] = torch.empty(G.info["n"], dtype=torch.int32, device="cuda")
        state["buf"] = torch.zeros((int(2 * _size(case)[1] * case["fraction"]) + 4096, 2),
                                   dtype=torch.int32, device="cuda")
    return state


def _sums(s):
    return dict(k=int(s.k), sum=np.array(s.sum).view(np.int64), sumsq=np.array(s.sumsq).view(np.int64))


def _result(r):
    return dict(x=np.array(r.x), var=np.array(r.var), lb=np.array(r.lb), ub=np.array(r.ub))


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "batch":
        b = state["batch"]
        got = b.count()
        raw = np.frombuffer(got, dtype=np.int64).reshape(b.num_graphs, -1)
        return dict(sums=raw)
    if op == "serve":
        srv = state["server"]
        tickets = [srv.submit(g, f, s, mask) for g, f, s, mask in state["requests"]]
        out = [srv.wait(t) for t in tickets]
        return dict(k=np.array([st["k"] for _, st in out]), x=np.array([list(r.x) for r, _ in out]),
                    var=np.array([list(r.var) for r, _ in out]))
    if op == "register":
        G = gs.Graph(state["row"], state["col"], hub_budget_bytes=state["budget"])
        s = G.count(None, gs.GS_THREE_NODE)
        info = [G.info["n"], G.info["m"], G.info["max_degree"]]
        G.close()
        return dict(info=np.array(info), est=_result(gs.gs_estimate(s)), **_sums(s))
    G = state["graph"]
    if op == "count" or op == "count3":
        s = G.count(None, gs.GS_CONNECTED if op == "count" else gs.GS_THREE_NODE)
        return dict(est=_result(gs.gs_estimate(s)), **_sums(s))
    if op == "estimate":
        r, k = G.count_estimate(case["fraction"], seed=state["seed"])
        return dict(k=k, est=_result(r))
    if op == "explicit":
        pairs = state["pairs"]
        per = torch.empty((pairs.shape[0], 3), dtype=torch.int64, device="cuda")
        conn = G.count(pairs, gs.GS_CONNECTED, per)
        disc = gs.gs_count_disconnected(G.handle, G.ws.handle, pairs, pairs.shape[0], per)
        return dict(per_edge=per, conn=_sums(conn), est=_result(gs.gs_estimate(conn)),
                    disc=_sums(disc), est_disc=_result(gs.gs_estimate_disconnected(disc)))
    if op == "micro":
        zmax, arg = gs.gs_micro(G.handle, G.ws.handle, state["pairs"], state["pairs"].shape[0],
                                case["p_e"], state["seed"], state["x"])
        return dict(x=state["x"], zmax=np.array(zmax), edge=np.array(arg))
    if op == "weighted":
        core, buf = state["core"], state["buf"]
        top = gs.gs_core_numbers(G.handle, G.ws.handle, core)
        k, s = gs.gs_sample_weighted(G.handle, G.ws.handle, core, case["fraction"], state["seed"],
                                     buf)
        r = gs.gs_count_weighted(G.handle, G.ws.handle, buf[:k], k, core, s)
        return dict(top=top, core=core, k=k, pairs=buf, scale=s, est=_result(r))
    if op == "adaptive":
        s, r, it, f = gs.gs_count_adaptive(G.handle, G.ws.handle, case["beta"], case["t_max"], 0.0,
                                           state["seed"])
        return dict(iters=it, fraction=f, est=_result(r), **_sums(s))
    raise ValueError(op)


# ------------------------------------------------------------------- work

def _size(case):
    """(vertices, edges) asked for."""
    if case["model"] == "rmat":
        n = 1 << case["scale"]
        # distinct edges: the generator's collisions grow with the scale's density
        return n, int(0.9 * n * case["edge_factor"])
    return case["n"], case["m"]


def work(case):
    """Bytes a pass cannot do without: the adjacency it is about, read once
    (whole for exact counts, the sampled edges' two lists at the mean degree of
    an edge's end for samples), and its outputs. Only integer work: no flops
    are counted."""
    op = case["op"]
    if op == "batch":
        n = case["count"] * (case["n_lo"] + case["n_hi"]) / 2
        m = n * (case["deg_lo"] + case["deg_hi"]) / 4
        return dict(bytes=8 * n + 8 * m + 272 * case["count"], flops=0)
    if op == "serve":
        f = (case["f_hi"] - case["f_lo"]) / math.log(case["f_hi"] / case["f_lo"])
        return dict(bytes=case["requests"] * f * 600000 * 400, flops=0)
    n, m = _size(case)
    whole = 8.0 * n + 8.0 * m
    if op in ("count", "count3", "register"):
        return dict(bytes=whole, flops=0)
    if op == "adaptive":
        return dict(bytes=min(whole, 2 * math.sqrt(m) * (16 + 8 * 20 * m / n)) + 264, flops=0)
    k = m * case["fraction"]
    lists = min(whole, k * (8 + 8 * 2 * m / n))
    if op == "micro":
        return dict(bytes=lists + 120 * k, flops=0)
    if op == "weighted":
        return dict(bytes=whole + 4 * n + 8 * k + lists, flops=0)
    return dict(bytes=lists + (24 * k if op == "explicit" else 264), flops=0)


# ------------------------------------------------------------------- 64 bits

def _mix(x):
    z = x + np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _keys(m, seed):
    with np.errstate(over="ignore"):
        return _mix(np.uint64(seed) ^ _mix(np.arange(m, dtype=np.uint64))) >> np.uint64(11)


def _contains(row, col, n, v, x):
    """x in N(v), elementwise."""
    keys = torch.repeat_interleave(torch.arange(n, device="cuda"), row[1:] - row[:-1]) * n + col
    q = v * n + x
    at = torch.searchsorted(keys, q).clamp_(max=max(keys.numel() - 1, 0))
    return keys[at] == q


def _oriented(row, pairs):
    """(u, v) with the lower degree first (ties: the smaller id)."""
    a, b = pairs[:, 0].long(), pairs[:, 1].long()
    deg = row[1:] - row[:-1]
    swap = (deg[a] > deg[b]) | ((deg[a] == deg[b]) & (a > b))
    return torch.where(swap, b, a), torch.where(swap, a, b)


def _triangles(row, col, u, v):
    n, deg, t = row.numel() - 1, row[1:] - row[:-1], torch.zeros_like(u)
    step = max(1, int(3e8 / max(1.0, float(deg[u].double().mean()))))
    for s in range(0, u.numel(), step):
        i, p = _expand(row[u[s:s + step]], deg[u[s:s + step]])
        hit = _contains(row, col, n, v[s:s + step][i], col[p].long())
        t[s:s + step] = torch.bincount(i[hit], minlength=t[s:s + step].numel())
    return t


def _counts(row, col, pairs):
    """Per edge (t, k, q, a, b): sparse products with 0/1 columns of T and S_v."""
    u, v = _oriented(row, pairs)
    n, deg = row.numel() - 1, row[1:] - row[:-1]
    A = torch.sparse_csr_tensor(row, col.long(), torch.ones(col.numel(), dtype=torch.float64, device="cuda"), (n, n))
    out = torch.zeros((u.numel(), 3), dtype=torch.int64, device="cuda")
    step = max(1, int(1.5e8 / n))
    for s in range(0, u.numel(), step):
        uu, vv = u[s:s + step], v[s:s + step]
        c = torch.arange(uu.numel(), device="cuda")
        nu = torch.zeros((n, uu.numel()), dtype=torch.float64, device="cuda")
        nv = torch.zeros_like(nu)
        for x, to in ((uu, nu), (vv, nv)):
            i, p = _expand(row[x], deg[x])
            to[col[p].long(), i] = 1.0
        T = nu * nv
        su, sv = nu - T, nv - T
        su[vv, c] = 0.0
        sv[uu, c] = 0.0
        out[s:s + step, 0] = T.sum(0).long()
        out[s:s + step, 1] = ((A @ T) * T).sum(0).long() // 2
        out[s:s + step, 2] = ((A @ sv) * su).sum(0).long()
    t = out[:, 0]
    return out, deg[u] - 1 - t, deg[v] - 1 - t


def _numerators(tkq, a, b):
    t, k, q = ([int(x) for x in tkq[:, j].tolist()] for j in range(3))
    rows = []
    for t, k, q, a, b in zip(t, k, q, a.tolist(), b.tolist()):
        n8 = t * (t - 1) // 2 - k
        rows.append((t, a + b, k, n8, t * (a + b) - 4 * n8, q,
                     a * (a - 1) + b * (b - 1) - t * (a + b) + 4 * n8, a * b - q))
    return rows


def _disconnected(rows, tkq, a, b, n, m):
    out = []
    for N, t, a, b in zip(rows, tkq[:, 0].tolist(), a.tolist(), b.tolist()):
        R = n - 2 - t - a - b
        c16 = m - (a + 1 + t) - (b + 1 + t) + 1
        n13 = 2 * t * R - N[4]
        n14 = (a + b) * R - 2 * N[7]
        n15 = c16 - N[2] - 4 * N[3] - N[4] - N[5] - 2 * N[7]
        n16 = R * (R - 1) // 2 - n15
        n17 = 2 * N[2] + 12 * N[3] + 6 * N[4] + 3 * N[5] + 2 * N[6] + 12 * N[7] + 2 * n13 + 6 * n14 + 6 * n15 + 12 * n16
        out.append((R, 2 * t + 3 * (a + b) + 6 * R, n13, n14, n15, n16, n17))
    return out


def _estimates(rows, m, den, total=None):
    """x, var, lb, ub of the expansion estimator from per-edge numerators."""
    K = len(rows)
    x, var = [], []
    for i, d in enumerate(den):
        s, s2 = sum(r[i] for r in rows), sum(r[i] * r[i] for r in rows)
        X = Fraction(m * s, K * d)
        x.append(float(total[i] - X if total and total[i] is not None else X))
        if K == m:
            var.append(0.0)
        elif K < 2:
            var.append(math.nan)
        else:
            var.append(float(Fraction(m * (m - K) * (K * s2 - s * s), K * K * (K - 1) * d * d)))
    x, var = np.array(x), np.array(var)
    return dict(x=x, var=var, lb=x - 1.96 * np.sqrt(var), ub=x + 1.96 * np.sqrt(var))


_NO_SUMS = dict(k=None, sum=None, sumsq=None)


def _cores(row, col):
    n = row.numel() - 1
    deg, core = row[1:] - row[:-1], torch.zeros(n, dtype=torch.int64, device="cuda")
    alive = torch.ones(n, dtype=torch.bool, device="cuda")
    k = 0
    while bool(alive.any()):
        k = max(k, int(deg[alive].min()))
        while True:
            out = torch.nonzero(alive & (deg <= k)).squeeze(1)
            if out.numel() == 0:
                break
            core[out], alive[out] = k, False
            _, p = _expand(row[out], (row[1:] - row[:-1])[out])
            deg = deg - torch.bincount(col[p].long(), minlength=n)
    return core


def _micro(case, seed, row, col, pairs):
    """Algorithm 7's rows by expanding every probe."""
    n, m, pe = row.numel() - 1, col.numel() // 2, case["p_e"]
    deg = row[1:] - row[:-1]
    u, v = _oriented(row, pairs)
    x = torch.zeros((u.numel(), 15), dtype=torch.float64, device="cuda")
    adj = torch.repeat_interleave(torch.arange(n, device="cuda"), deg) * n + col

    def has(y, z):
        q = y * n + z
        return adj[torch.searchsorted(adj, q).clamp_(max=adj.numel() - 1)] == q

    with np.errstate(over="ignore"):
        key = (np.minimum(u.cpu().numpy(), v.cpu().numpy()).astype(np.uint64) << np.uint64(32)) | np.maximum(u.cpu().numpy(), v.cpu().numpy()).astype(np.uint64)
        ekey = _mix(np.uint64(seed) ^ _mix(key))
    mean = float((deg[u] + deg[v]).double().mean())
    step = max(1, int(2e8 / (mean * (1 + pe * float((deg.double() ** 2).sum() / deg.sum())))))
    for s in range(0, u.numel(), step):
        uu, vv = u[s:s + step], v[s:s + step]
        c = uu.numel()
        iu, pu = _expand(row[uu], deg[uu])
        iv, pv = _expand(row[vv], deg[vv])
        wu, wv = col[pu].long(), col[pv].long()
        tu, tv = has(vv[iu], wu), has(uu[iv], wv)
        keep_u, keep_v = wu != vv[iu], (wv != uu[iv]) & ~tv
        e = torch.cat((iu[keep_u], iv[keep_v]))
        w = torch.cat((wu[keep_u], wv[keep_v]))
        cls = torch.cat((torch.where(tu[keep_u], 1, 2), torch.full((int(keep_v.sum()),), 3, device="cuda")))
        t = torch.bincount(iu[keep_u & tu], minlength=c)
        cw = torch.ceil(deg[w].double() * pe).long()
        with np.errstate(over="ignore"):
            h = _mix(ekey[s:s + step][e.cpu().numpy()] ^ w.cpu().numpy().astype(np.uint64))
            d = deg[w].cpu().numpy().astype(np.uint64)
            # high word of the 64 x 64-bit product, d below 2^31
            o = ((h >> np.uint64(32)) * d + (((h & np.uint64(0xFFFFFFFF)) * d) >> np.uint64(32))) >> np.uint64(32)
        o = torch.as_tensor(o.astype(np.int64), device="cuda")
        i, j = _expand(o, cw)
        j = torch.where(j >= deg[w[i]], j - deg[w[i]], j)
        r, ee, ww, cc = col[row[w[i]] + j].long(), e[i], w[i], cls[i]
        inu, inv, above = has(uu[ee], r), has(vv[ee], r), r > ww
        end = (r == uu[ee]) | (r == vv[ee])
        wt = deg[ww].double() / cw[i].double()
        four = (cc == 1) & inu & inv & above
        om = (cc != 1) & ~end & inu & inv
        cyc = (cc == 2) & ~end & inv & ~inu
        tail = ~end & above & (((cc == 2) & inu & ~inv) | ((cc == 3) & inv & ~inu))
        tot = [torch.zeros(c, dtype=torch.float64, device="cuda").index_add_(0, ee[z], wt[z])
               for z in (four, tail, cyc, om)]
        a, b = deg[uu] - 1 - t, deg[vv] - 1 - t
        t, a, b = t.double(), a.double(), b.double()
        R = n - 2 - t - a - b
        f = x[s:s + step]
        n3 = Fraction(n * (n - 1) * (n - 2), 6) - (n - 2)
        cols = [t, a + b, R, torch.full_like(t, float(n3)), tot[0], t * (t - 1) / 2 - tot[0], tot[1], tot[2],
                a * (a - 1) / 2 + b * (b - 1) / 2 - tot[1], a * b - tot[2], t * R, (a + b) * R,
                m - (t + deg[uu] + deg[vv] + 1) - tot[3], R * (R - 1) / 2]
        for k, z in enumerate(cols):
            f[:, k] = z
        f[:, 14] = float(Fraction(n * (n - 1) * (n - 2) * (n - 3), 24)) - f[:, 4:14].sum(1)
    return x


def exact(case, seed):
    op = case["op"]
    if op in ("batch", "serve"):
        return None  # whole numbers; hundreds of graphs or requests
    n_ask, m_ask = _size(case)
    k_ask = m_ask * case.get("fraction", 4 * m_ask ** -0.5 if op == "adaptive" else 1.0)
    if op in ("count3", "register"):
        if m_ask > 3e6:
            return None
    elif op == "micro":
        if k_ask > 3e4 or m_ask > 3e6:
            return None
    elif k_ask * m_ask > 5e10 or k_ask * n_ask > 5e9:
        return None
    row, col = _csr(*_edges(case, _gen(seed)))
    n, m = n_ask, col.numel() // 2
    seed64 = int(seed) & (2**63 - 1)
    up = _upper(row, col)
    if op in ("count3", "register"):
        u, v = _oriented(row, up)
        t = _triangles(row, col, u, v)
        deg = row[1:] - row[:-1]
        # the other graphlets are not asked for: their fields are NaN
        x = [float(Fraction(int(t.sum()), 3)), float(Fraction(int((deg[u] + deg[v] - 2 - 2 * t).sum()), 2))]
        z, zero = np.full(8, np.nan), np.full(8, np.nan)
        z[:2], zero[:2] = x, 0.0
        est = dict(x=z, var=zero, lb=z, ub=z)
        got = dict(est=est, **_NO_SUMS)
        return dict(info=None, **got) if op == "register" else got
    if op == "count":
        return dict(est=_estimates(_numerators(*_counts(row, col, up)), m, D), **_NO_SUMS)
    if op == "estimate":
        keep = _keys(m, seed64) < np.uint64(math.floor(case["fraction"] * 2.0**53))
        pairs = up[torch.as_tensor(keep, device="cuda")]
        if pairs.shape[0] < 2:
            return None
        return dict(k=None, est=_estimates(_numerators(*_counts(row, col, pairs)), m, D))
    if op == "explicit" or op == "micro":
        pairs = _sample(case, seed, row, col)
        if pairs.shape[0] < 2:
            return None
        if op == "micro":
            x = _micro(case, seed64, row, col, pairs)
            return dict(x=x, zmax=x.max(0).values, edge=None)
        tkq, a, b = _counts(row, col, pairs)
        rows = _numerators(tkq, a, b)
        disc = _disconnected(rows, tkq, a, b, n, m)
        c3, c4 = Fraction(n * (n - 1) * (n - 2), 6), Fraction(n * (n - 1) * (n - 2) * (n - 3), 24)
        return dict(per_edge=None, conn=_NO_SUMS, est=_estimates(rows, m, D), disc=_NO_SUMS,
                    est_disc=_estimates(disc, m, D_DISC, [None, c3, None, None, None, None, c4]))
    if op == "weighted":
        core = _cores(row, col)
        we = torch.minimum(core[up[:, 0].long()], core[up[:, 1].long()])
        W = int(we.sum())
        if W == 0:
            return None
        scale = case["fraction"] * m / W
        pi = np.minimum(1.0, scale * we.cpu().numpy().astype(np.float64))
        keep = _keys(m, seed64) < np.floor(pi * 2.0**53).astype(np.uint64)
        pairs, pi = up[torch.as_tensor(keep, device="cuda")], pi[keep]
        rows = np.array(_numerators(*_counts(row, col, pairs)), dtype=np.float64)
        x = (rows / pi[:, None]).sum(0) / np.array(D)
        var = ((1 - pi)[:, None] * (rows / pi[:, None]) ** 2).sum(0) / np.array(D, dtype=np.float64) ** 2
        est = dict(x=x, var=var, lb=x - 1.96 * np.sqrt(var), ub=x + 1.96 * np.sqrt(var))
        return dict(top=None, core=None, k=None, pairs=None, scale=scale, est=est)
    if op == "adaptive":
        order = np.argsort(_keys(m, seed64), kind="stable")
        J, phi, prev, rows, loss, it = 0, 1.0 / math.sqrt(m), None, [], 1.0, 0
        while loss > case["beta"] and it < case["t_max"]:
            new = min(m, J + math.ceil(phi * (m - J)))
            if (new * 1.0) * m > 2e11 or new * n > 2e10:
                return None
            if new > J:
                rows += _numerators(*_counts(row, col, up[torch.as_tensor(order[J:new], device="cuda")]))
            J, phi, it = new, phi / 2, it + 1
            est = _estimates(rows, m, D)
            if prev is not None:
                loss = max((0.0 if y == p else math.inf if p == 0 else abs(y - p) / abs(p))
                           for y, p in zip(est["x"][2:], prev[2:]))
            prev = est["x"]
        return dict(iters=None, fraction=J / m, est=est, **_NO_SUMS)
    return None

"""The work a user of this library has it do, as cases that can be timed.

Sizes and shapes are those of the benchmark's workloads, of its batched and
served forms and of the tests: bipartite transaction graphs with Zipf(1.8)
items, undirected R-MAT graphs (0.57, 0.19, 0.19), a planted block, the
clique metrics on small R-MAT graphs.  Inputs are drawn on the GPU from the
seed; a state holds the resident graph handles, result buffers or the server
that a caller keeps, and one pass is one call (or one burst of requests) with
all its results.
"""
import math

import numpy as np
import torch

from paper_2504_09311_gb300 import dupin

Q_ONE = 1 << 32
ZIPF = 1.8


def listed():
    return [
        # a plug-in's smallest request: one window of 1,000 transactions in buffers the caller owns
        {"name": "noalloc_1k", "kind": "noalloc", "edges": 1000, "metric": "fd", "k": 1, "lpo": False},
        # one mid-size graph through the plain call with host results (the small DG workload)
        {"name": "block_dg", "kind": "block", "users": 10_000, "metric": "dg", "k": 1, "lpo": False},
        # a serving-sized batch of transaction windows, fewer graphs than the GPU has places for
        {"name": "windows_61", "kind": "windows", "count": 61, "k": 1},
        # the batched workload: thousands of uneven windows in one call
        {"name": "windows_4096", "kind": "windows", "count": 4096, "k": 1},
        # a burst of served requests over resident windows, one large graph among them
        {"name": "serve_40", "kind": "serve", "requests": 40, "scale": 18},
        # one transaction graph of 40M edges under three eps, as a parameter search runs it
        {"name": "zipf_3eps", "kind": "zipf", "users": 2_000_000, "per_user": 20, "k": 1},
        # the headline: FD and DG peels of R-MAT scale 24 in one call, thousands of rounds each
        {"name": "rmat24_fd_dg", "kind": "rmat", "scale": 24, "metrics": "fd,dg", "k": 1, "lpo": False},
        # the paper's setting k = 2: few rounds, all over the whole graph
        {"name": "rmat24_fd_k2", "kind": "rmat", "scale": 24, "metrics": "fd", "k": 2, "lpo": False},
        # weighted edges and vertices with the paper's local trims (Algorithm 4)
        {"name": "rmat21_dw_lpo", "kind": "rmat", "scale": 21, "metrics": "dw", "k": 1, "lpo": True},
        # a new graph for every call: load from page-locked host memory, validate, peel, copy back, free
        {"name": "load_zipf_8m", "kind": "load", "users": 500_000, "per_user": 16, "k": 2},
        # triangle density
        {"name": "tds_rmat15", "kind": "clique", "scale": 15, "q": 3, "k": 3},
        # 4-clique density
        {"name": "kclids4_rmat13", "kind": "clique", "scale": 13, "q": 4, "k": 4},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["noalloc", "block", "windows", "serve", "zipf", "rmat", "rmat", "load", "clique"])
    k = rng.choice([1, 1, 2])
    if kind == "noalloc":
        return {"kind": kind, "edges": log_int(1000, 50_000), "metric": rng.choice(["fd", "dg"]), "k": k,
                "lpo": rng.random() < 0.25}
    if kind == "block":
        return {"kind": kind, "users": log_int(1500, 60_000), "metric": rng.choice(["dg", "dw"]), "k": k,
                "lpo": rng.random() < 0.25}
    if kind == "windows":
        return {"kind": kind, "count": log_int(8, 4000), "k": k}
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(8, 48), "scale": rng.randint(17, 20)}
    if kind == "zipf":
        return {"kind": kind, "users": log_int(150_000, 1_900_000), "per_user": rng.randint(8, 20), "k": k}
    if kind == "load":
        return {"kind": kind, "users": log_int(20_000, 900_000), "per_user": rng.randint(8, 18), "k": k}
    if kind == "clique":
        q = rng.choice([3, 3, 4, 5])
        if q == 3 and rng.random() < 0.3:  # one vertex at a time: hundreds of rounds
            return {"kind": kind, "scale": rng.randint(9, 12), "q": 3, "k": 1}
        return {"kind": kind, "scale": rng.randint(9, {3: 15, 4: 13, 5: 11}[q]), "q": q, "k": q}
    return {"kind": kind, "scale": rng.randint(17, 23), "metrics": rng.choice(["fd", "dg", "dw", "fd,dg"]), "k": k,
            "lpo": rng.random() < 0.2}


# ------------------------------------------------------------------ inputs


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _distinct(keys):
    keys = torch.sort(keys).values
    if keys.numel() < 2:
        return keys
    first = torch.ones_like(keys, dtype=torch.bool)
    first[1:] = keys[1:] != keys[:-1]
    return keys[first]


def _ptr(sorted_rows, n):
    return torch.searchsorted(sorted_rows, torch.arange(n + 1, device="cuda", dtype=sorted_rows.dtype))


def _fd(deg):
    """Fraudar's 1 / ln(degree + 5) in Q32.32."""
    return (Q_ONE / torch.log(deg.double() + 5.0)).long()


def _hash(x, seed):
    x = (x ^ (seed * 0x632BE5AB)) * 0x9E3779B97F4A7C1
    x = (x ^ (x >> 29)) * 0x1B873593CC9E2D51
    return (x ^ (x >> 32)) & 0x7FFFFFFF


def _zipf_cdf(n):
    return torch.cumsum(torch.arange(1, n + 1, device="cuda", dtype=torch.float64) ** -ZIPF, 0)


def _zipf_draws(users, edges):
    """Draws after which about 'edges' distinct (user, Zipf item) pairs have come up."""
    return int(1.88 * (edges / (2.01 * users)) ** ZIPF * users) + 64


def _bipartite(users, items, per_user, seed, blocks=0):
    """Distinct (user, item) keys: users uniform, items Zipf over a permutation, and planted blocks
    of up to 500 x 500 pairs (p = 0.3) with 150 camouflage pairs per block user."""
    g = _gen(seed)
    d = _zipf_draws(users, users * per_user)
    cdf = _zipf_cdf(items)
    rank = torch.searchsorted(cdf, torch.rand(d, generator=g, device="cuda", dtype=torch.float64) * cdf[-1])
    perm = torch.randperm(items, generator=g, device="cuda")
    keys = [(torch.randint(users, (d,), generator=g, device="cuda") << 32) | perm[rank.clamp_(max=items - 1)]]
    for _ in range(blocks):
        bu = torch.randperm(users, generator=g, device="cuda")[: min(500, users)]
        bi = torch.randperm(items, generator=g, device="cuda")[: min(500, items)]
        full = ((bu[:, None] << 32) | bi[None, :]).reshape(-1)
        keys.append(full[torch.rand(full.numel(), generator=g, device="cuda") < 0.3])
        keys.append(((bu[:, None] << 32) | torch.randint(items, (bu.numel(), 150), generator=g, device="cuda")).reshape(-1))
    return _distinct(torch.cat(keys))


def _block(users, seed):
    """users x users/2 with 10 uniform pairs per user and a planted 200 x 200 block at p = 0.5."""
    g = _gen(seed)
    items = users // 2
    d = 10 * users
    keys = (torch.randint(users, (d,), generator=g, device="cuda") << 32) | torch.randint(items, (d,), generator=g, device="cuda")
    bu = torch.randperm(users, generator=g, device="cuda")[:200]
    bi = torch.randperm(items, generator=g, device="cuda")[:200]
    full = ((bu[:, None] << 32) | bi[None, :]).reshape(-1)
    full = full[torch.rand(full.numel(), generator=g, device="cuda") < 0.5]
    return _distinct(torch.cat([keys, full]))


def _csr_csc(keys, users, items, metric, seed):
    """(csr_ptr, csr_idx, csr_w, csc_ptr, csc_idx, csc_w) of sorted (user << 32 | item) keys."""
    u, i = keys >> 32, keys & 0xFFFFFFFF
    back = torch.sort((i << 32) | u).values
    bi, bu = back >> 32, back & 0xFFFFFFFF
    csr_ptr, csc_ptr = _ptr(u, users), _ptr(bi, items)
    w = wb = None
    if metric == "fd":
        by_item = _fd(csc_ptr[1:] - csc_ptr[:-1])
        w, wb = by_item[i], by_item[bi]
    elif metric == "dw":
        w = (1 + _hash(keys, seed) % 100) << 32
        wb = (1 + _hash((bu << 32) | bi, seed) % 100) << 32
    return csr_ptr, i.int(), w, csc_ptr, bu.int(), wb


def _rmat(scale, seed):
    """Distinct (u << 32 | v) keys with both directions of every edge, sorted: an undirected R-MAT
    graph of 2^scale relabelled vertices, 16 draws per vertex, self-loops dropped."""
    g = _gen(seed)
    n = 1 << scale
    d = 16 * n
    u = torch.zeros(d, dtype=torch.int64, device="cuda")
    v = torch.zeros(d, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        r = torch.rand(d, generator=g, device="cuda")
        u.mul_(2).add_(r >= 0.76)
        v.mul_(2).add_(((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    perm = torch.randperm(n, generator=g, device="cuda")
    u, v = perm[u], perm[v]
    u, v = u[u != v], v[u != v]
    key = _distinct((torch.minimum(u, v) << 32) | torch.maximum(u, v))
    del u, v
    return torch.sort(torch.cat([key, ((key & 0xFFFFFFFF) << 32) | (key >> 32)])).values


def _rmat_csr(scale, weights, seed):
    """(n, ptr, idx, w, a): weights 'fd' (by the larger end's degree), 'dw' (1..100, a in 0..10) or none."""
    n = 1 << scale
    key = _rmat(scale, seed)
    u, v = key >> 32, key & 0xFFFFFFFF
    ptr = _ptr(u, n)
    w = a = None
    if weights == "fd":
        w = _fd(ptr[1:] - ptr[:-1])[torch.maximum(u, v)]
    elif weights == "dw":
        w = (1 + _hash((torch.minimum(u, v) << 32) | torch.maximum(u, v), seed) % 100) << 32
        a = torch.randint(11, (n,), generator=_gen(seed + 1), device="cuda") << 32
    return n, ptr, v.int(), w, a


def _window_sizes(count):
    """Edges per window: log-uniform in 1,000 .. 500,000, multiples of 1,000."""
    r = np.random.RandomState(count).uniform(math.log(1000), math.log(500_000), count)
    return np.maximum(1000, np.round(np.exp(r) / 1000).astype(np.int64) * 1000)


def _windows(sizes, seed):
    """A resident graph per size m: m/10 users x m/20 items, about m Zipf pairs, Fraudar weights."""
    graphs = []
    at = 0
    cdf = _zipf_cdf(int(sizes.max()) // 20)
    while at < len(sizes):  # groups of about 2^28 draws
        end, draws = at, 0
        while end < len(sizes) and (end == at or draws < 1 << 28):
            draws += _zipf_draws(sizes[end] / 10, sizes[end])
            end += 1
        m = sizes[at:end]
        nu, ni = m // 10, m // 20
        dr = np.array([_zipf_draws(x / 10, x) for x in m], np.int64)
        g = _gen(seed * 131 + at)
        dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
        w = torch.repeat_interleave(torch.arange(len(m), device="cuda"), dev(dr))
        nut, nit = dev(nu), dev(ni)
        top = cdf[nit - 1]
        item = torch.searchsorted(cdf, torch.rand(w.numel(), generator=g, device="cuda", dtype=torch.float64) * top[w])
        item = (torch.minimum(item, nit[w] - 1) * 1_000_003 + 12_345) % nit[w]
        user = (torch.rand(w.numel(), generator=g, device="cuda", dtype=torch.float64) * nut[w]).long()
        key = _distinct((w << 40) | (user << 20) | item)
        w, user, item = key >> 40, (key >> 20) & 0xFFFFF, key & 0xFFFFF
        first = _ptr(w, len(m))
        back = torch.sort((w << 40) | (item << 20) | user).values
        uo, io = np.concatenate([[0], np.cumsum(nu + 1)]), np.concatenate([[0], np.cumsum(ni + 1)])

        def ptrs(keys, off, cnt):  # the windows' offset arrays end to end, each from 0
            k = torch.repeat_interleave(torch.arange(len(m), device="cuda"), dev(cnt + 1))
            j = torch.arange(k.numel(), device="cuda") - dev(off[:-1])[k]
            return torch.searchsorted(keys, (k << 40) | (j << 20)) - first[k]

        cp, rp = ptrs(key, uo, nu), ptrs(back, io, ni)
        deg = torch.zeros_like(rp)
        deg[:-1] = rp[1:] - rp[:-1]
        fd, iot = _fd(deg.clamp_(min=0)), dev(io[:-1])
        cw, rw = fd[iot[w] + item], fd[iot[back >> 40] + ((back >> 20) & 0xFFFFF)]
        ci, ri = item.int(), (back & 0xFFFFF).int()
        f = first.tolist()
        for j in range(len(m)):
            s, e = f[j], f[j + 1]
            graphs.append(dupin.Graph.load_bipartite(
                int(nu[j]), int(ni[j]), cp[uo[j]:uo[j + 1]], ci[s:e], cw[s:e], rp[io[j]:io[j + 1]], ri[s:e], rw[s:e],
                device_ptrs=True))
        at = end
    return graphs


def _flags(case):
    return dupin.LPO if case.get("lpo") else 0


EPS = (1, 10)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        m = case["edges"]
        users, items = m // 10, m // 20
        keys = _bipartite(users, items, 10, seed)
        cp, ci, cw, rp, ri, rw = _csr_csc(keys, users, items, "fd", seed)
        n = users + items
        s = {"n": n, "ptr": torch.cat([cp, rp[1:] + keys.numel()]), "idx": torch.cat([ci + users, ri]),
             "w": torch.cat([cw, rw]), "params": dupin.make_params(case["metric"], case["k"], EPS, flags=_flags(case)),
             "round": torch.empty(n, dtype=torch.int32, device="cuda"),
             "mask": torch.empty(n, dtype=torch.uint8, device="cuda"),
             "trace": [torch.zeros(n + 2, dtype=torch.int64, device="cuda") for _ in range(4)]}
    elif kind == "block":
        keys = _block(case["users"], seed)
        s = {"graph": _load(case["users"], case["users"] // 2, _csr_csc(keys, case["users"], case["users"] // 2, case["metric"], seed))}
    elif kind == "windows":
        graphs = _windows(_window_sizes(case["count"]), seed)
        s = {"graphs": graphs, "params": [dupin.make_params("fd", case["k"], EPS)] * len(graphs),
             "buffers": dupin.BatchBuffers.for_graphs(graphs, want_rounds=True, pinned=True)}
    elif kind == "serve":
        graphs = _windows(_window_sizes(case["requests"] - 1), seed)
        n, ptr, idx, w, a = _rmat_csr(case["scale"], "fd", seed)
        graphs.insert(len(graphs) // 2, dupin.Graph.load_symmetric(n, ptr, idx, w, a, device_ptrs=True))
        s = {"graphs": graphs, "params": dupin.make_params("fd", 1, EPS),
             "server": dupin.Server(memory_budget=16 << 30, max_slots=8)}
    elif kind == "zipf":
        users, items = case["users"], case["users"] // 2
        keys = _bipartite(users, items, case["per_user"], seed, blocks=5)
        g = _load(users, items, _csr_csc(keys, users, items, "fd", seed))
        s = {"graphs": [g] * 3, "params": [dupin.make_params("fd", case["k"], e) for e in ((0, 1), (1, 20), (1, 5))]}
        _device_results(s, g.n, 3)
    elif kind == "rmat":
        metrics = case["metrics"].split(",")
        n, ptr, idx, w, a = _rmat_csr(case["scale"], metrics[0], seed)
        g = dupin.Graph.load_symmetric(n, ptr, idx, w, a, device_ptrs=True)
        s = {"graphs": [g] * len(metrics), "params": [dupin.make_params(x, case["k"], EPS, flags=_flags(case)) for x in metrics]}
        _device_results(s, n, len(metrics))
    elif kind == "load":
        users, items = case["users"], case["users"] // 2
        keys = _bipartite(users, items, case["per_user"], seed, blocks=5)
        host = [x.cpu().pin_memory().numpy() for x in _csr_csc(keys, users, items, "fd", seed)]
        s = {"users": users, "items": items, "host": host, "params": [dupin.make_params("fd", case["k"], EPS)],
             "buffers": [dupin.result_buffers(users + items, True, True, True, pinned=True)]}
        for t in s["buffers"][0][2]:
            t[:] = 0
    else:
        n, ptr, idx, _, _ = _rmat_csr(case["scale"], "dg", seed)
        s = {"graph": dupin.Graph.load_symmetric(n, ptr, idx, device_ptrs=True)}
    s["case"] = case
    torch.cuda.empty_cache()  # the library allocates beside torch
    return s


def _load(users, items, arrays):
    return dupin.Graph.load_bipartite(users, items, *arrays, device_ptrs=True)


def _device_results(s, n, k):
    s["rounds"] = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(k)]
    s["masks"] = [torch.empty(n, dtype=torch.uint8, device="cuda") for _ in range(k)]


# ------------------------------------------------------------------ passes


def _numbers(results):
    """Rounds, best round, best size, best f (two words) and minimum-rule rounds of each peel."""
    return np.array([[r.n_rounds, r.best_round, r.best_size, r.best_f >> 32, r.best_f & 0xFFFFFFFF, r.n_min_rule]
                     for r in results], np.int64)


def _struct_numbers(results):
    f = [(int(r.best_f_hi) << 64) + int(r.best_f_lo) for r in results]
    return np.array([[r.n_rounds, r.best_round, r.best_size, x >> 32, x & 0xFFFFFFFF, r.n_min_rule]
                     for r, x in zip(results, f)], np.int64)


def _density(results):
    return np.array([r.best_density for r in results], np.float64)


def _host_output(o):
    # the trace arrays in their full length (zero after the last round): the same shape for every input
    f_hi, f_lo, size, peeled = (t.base for t in (o.trace_f_hi, o.trace_f_lo, o.trace_size, o.trace_peeled))
    return {"round": o.peel_round, "mask": o.best_mask, "f_hi": f_hi, "f_lo": f_lo.view(np.int64), "size": size,
            "peeled": peeled, "numbers": _numbers([o]), "density": _density([o])}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "noalloc":
        r = dupin.peel_noalloc(state["n"], state["ptr"], state["idx"], state["w"], None, state["params"], state["round"],
                               state["mask"], state["trace"])
        return {"round": state["round"], "mask": state["mask"], "trace": state["trace"],
                "numbers": _struct_numbers([r]), "density": _density([r])}
    if kind == "block":
        return _host_output(dupin.peel(state["graph"], case["metric"], case["k"], EPS, flags=_flags(case)))
    if kind == "clique":
        if case["q"] == 3:
            return _host_output(dupin.peel(state["graph"], "tds", case["k"], EPS))
        return _host_output(dupin.peel(state["graph"], "kclids", case["k"], EPS, clique_q=case["q"]))
    if kind == "windows":
        outs = dupin.peel_batch(state["graphs"], state["params"], buffers=state["buffers"])
        return {"rounds": state["buffers"]._block, "numbers": _numbers(outs), "density": _density(outs)}
    if kind == "serve":
        srv = state["server"]
        tickets = [srv.submit(g, state["params"]) for g in state["graphs"]]
        outs = [srv.wait(t) for t in tickets]
        return {"rounds": [o.peel_round for o in outs], "numbers": _numbers(outs), "density": _density(outs)}
    if kind == "load":
        g = dupin.Graph.load_bipartite(state["users"], state["items"], *state["host"])
        o = dupin.peel_batch([g], state["params"], want_rounds=True, want_trace=True, want_mask=True,
                             buffers=state["buffers"])[0]
        g.free()
        return _host_output(o)
    if len(state["graphs"]) == 1:
        r = [dupin.peel_device(state["graphs"][0], state["params"][0], state["rounds"][0], state["masks"][0])]
    else:
        r = dupin.peel_batch_device(state["graphs"], state["params"], state["rounds"], state["masks"])
    return {"rounds": state["rounds"], "masks": state["masks"], "numbers": _struct_numbers(r), "density": _density(r)}


# ------------------------------------------------------------------ work


def _graph_bytes(n, arcs, weighted, vertex=False):
    return 8 * (n + 1) + arcs * (12 if weighted else 4) + (8 * n if vertex else 0)


def work(case):
    """The adjacency (offsets, ids, weights) read once and each vertex's round and mask written once;
    one subtraction per arc.  Edge counts are the nominal ones."""
    kind = case["kind"]
    if kind == "noalloc":
        n, arcs = case["edges"] // 10 + case["edges"] // 20, 2 * case["edges"]
        b = _graph_bytes(n, arcs, case["metric"] != "dg") + 5 * n
    elif kind == "block":
        n, arcs = case["users"] + case["users"] // 2, 2 * (10 * case["users"] + 20_000)
        b = _graph_bytes(n, arcs, case["metric"] != "dg") + 5 * n
    elif kind in ("windows", "serve"):
        count = case["count"] if kind == "windows" else case["requests"] - 1
        m = int(count * 499_000 / math.log(500))  # the mean of the log-uniform sizes
        n, arcs = 3 * m // 20, 2 * m
        b = _graph_bytes(n, arcs, True) + 4 * n
        if kind == "serve":
            b += _graph_bytes(1 << case["scale"], 32 << case["scale"], True) + (4 << case["scale"])
            arcs += 32 << case["scale"]
    elif kind in ("zipf", "load"):
        n, arcs = case["users"] + case["users"] // 2, 2 * case["users"] * case["per_user"]
        peels = 3 if kind == "zipf" else 1
        b = _graph_bytes(n, arcs, True) + 5 * n * peels
        arcs *= peels
    elif kind == "rmat":
        metrics = case["metrics"].split(",")
        n, arcs = 1 << case["scale"], 32 << case["scale"]
        b = _graph_bytes(n, arcs, metrics[0] != "dg", metrics[0] == "dw") + 5 * n * len(metrics)
        arcs *= len(metrics)
    else:
        n, arcs = 1 << case["scale"], 32 << case["scale"]
        b = _graph_bytes(n, arcs, False) + 5 * n
        arcs *= 32  # listing: each arc's two rows are merged, about a row's length of comparisons
    return {"bytes": b, "flops": arcs}


# ------------------------------------------------------------------ exact values


def _whole_sum(x):
    return (int((x >> 32).sum()) << 32) + int((x & 0xFFFFFFFF).sum())


def _best_density(ptr, idx, w, k, eps):
    """The best prefix's density of Algorithm 2 (threshold k (1 + eps) g, the minimum rule where it
    selects nobody), in whole numbers."""
    n = len(ptr) - 1
    row = np.repeat(np.arange(n), np.diff(ptr))
    wt = np.zeros(n, np.int64)
    np.add.at(wt, row, w)
    f = _whole_sum(wt) // 2
    best = (f, n)
    live = np.arange(n)
    alive = np.ones(n, bool)
    leaving = np.zeros(n, bool)
    while len(live):
        cur = wt[live]
        sel = cur <= min(k * (eps[1] + eps[0]) * f // (eps[1] * len(live)), (1 << 63) - 1)
        if not sel.any():
            sel = cur == cur.min()
        out, live = live[sel], live[~sel]
        leaving[out] = True
        alive[out] = False
        arcs = np.concatenate([np.arange(ptr[u], ptr[u + 1]) for u in out])
        heads, c = idx[arcs], w[arcs]
        f -= _whole_sum(cur[sel]) - _whole_sum(c[leaving[heads]]) // 2
        np.subtract.at(wt, heads[alive[heads]], c[alive[heads]])
        leaving[out] = False
        if len(live) and f * best[1] > best[0] * len(live):
            best = (f, len(live))
    return best[0] / Q_ONE / best[1]


def exact(case, seed):
    """The best density of the single peels that a plain loop over rounds settles quickly; every other
    output is a whole number."""
    if case["kind"] not in ("noalloc", "block") or case.get("lpo") or case.get("users", 0) > 20_000:
        return None
    if case["kind"] == "noalloc":
        users, items = case["edges"] // 10, case["edges"] // 20
        keys = _bipartite(users, items, 10, seed)
        arrays = _csr_csc(keys, users, items, "fd", seed)
    else:
        users, items = case["users"], case["users"] // 2
        keys = _block(users, seed)
        arrays = _csr_csc(keys, users, items, case["metric"], seed)
    cp, ci, cw, rp, ri, rw = [None if x is None else x.cpu().numpy() for x in arrays]
    ptr = np.concatenate([cp, rp[1:] + len(ci)])
    idx = np.concatenate([ci + users, ri])
    w = np.full(len(idx), Q_ONE, np.int64) if case["metric"] == "dg" else np.concatenate([cw, rw])
    return {"density": np.array([_best_density(ptr, idx, w, case["k"], EPS)])}

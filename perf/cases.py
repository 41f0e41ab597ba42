"""Workloads of the library as a program runs them: one pass of each through the public entry points.

`listed()` are the named workloads, `draw(rng)` more of the same ranges; `prepare` makes what a program has
before the call (descriptors, a graph, eigenpairs, a server), `run` is one call, `exact` the same result in
fp64 torch without the library, `work` the bytes and operations no implementation can do without.

Not here: the eigendecomposition, SHybrid sparsification and spectrum bounds, which run once per database and
spend their time in cuBLAS / cuSOLVER or in a single pass; general transfer functions and the paper's two
other solver forms, which run the same products as the query cases.
"""
import math

import numpy as np
import torch

import paper_1807_08692_gb300 as hd

ALPHA = 0.99
GAMMA = 3.0
P_IN = 0.4          # share of a node's edges inside its own cluster
HALF_DEGREE = 27    # edges a node picks (the union of both ends' picks has about twice as many per row)


def listed():
    return [
        # the workload of the unit-sized configuration: 2,000 nodes, 16 queries, rank 50; bound by latency
        {"name": "query_2k_b16", "kind": "query", "n": 2000, "B": 16, "r": 50, "storage": "bf16", "tol": 3e-4, "k_y": 10},
        # 100,000 nodes, an odd batch, compact (fp8) eigenvectors and the recipes' tight tolerance
        {"name": "query_100k_b37_fp8", "kind": "query", "n": 100000, "B": 37, "r": 100, "storage": "fp8", "tol": 1e-6, "k_y": 50},
        # one interactive query on the million-node database
        {"name": "query_1m_b1", "kind": "query", "n": 1000000, "B": 1, "r": 200, "storage": "bf16", "tol": 3e-4, "k_y": 10},
        # the headline: 64 queries per batch, hybrid with 200 eigenpairs in bf16
        {"name": "query_1m_b64", "kind": "query", "n": 1000000, "B": 64, "r": 200, "storage": "bf16", "tol": 3e-4, "k_y": 10},
        # the largest batch of the sweep without eigenpairs (plain conjugate gradient)
        {"name": "cg_1m_b256", "kind": "query", "n": 1000000, "B": 256, "r": 0, "storage": "bf16", "tol": 3e-4, "k_y": 10},
        # top-100 of a batch's scores
        {"name": "rank_1m_b64", "kind": "rank", "n": 1000000, "B": 64, "K": 100, "pool": 0},
        # observations of a batch of query descriptors (the first online step): fp32 and bf16 databases
        {"name": "observe_100k_f32", "kind": "observe", "n": 100000, "d": 512, "nq": 64, "k_y": 50, "dtype": "f32"},
        {"name": "observe_1m_bf16", "kind": "observe", "n": 1000000, "d": 2048, "nq": 64, "k_y": 10, "dtype": "bf16"},
        # indexing a database: the k-NN graph, fp32 (the 100,000-node configuration) and bf16 descriptors
        {"name": "graph_100k_f32", "kind": "graph", "n": 100000, "d": 512, "k": 50, "dtype": "f32"},
        {"name": "graph_250k_bf16", "kind": "graph", "n": 250000, "d": 512, "k": 50, "dtype": "bf16"},
        # a saturated server: mixed tolerances and K, twice as many requests as slots
        {"name": "serve_1m", "kind": "serve", "n": 1000000, "slots": 128, "requests": 256, "r": 200, "storage": "bf16"},
        # truncated temporal filtering at the setting of the paper's Table 1: 75,000-item shortlists, 20 iterations
        {"name": "truncated_1m_b64", "kind": "truncated", "n": 1000000, "B": 64, "s": 75000, "iters": 20, "k_y": 10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "query", "rank", "observe", "graph", "serve", "truncated"])
    n = _log_int(rng, 2000, 1000000)
    if kind == "query":
        r = min(rng.choice([0, 1, 50, 100, 200, 400]), n // 20)
        return {"kind": kind, "n": n, "B": _log_int(rng, 1, 256), "r": r,
                "storage": rng.choice(["f32", "bf16", "bf16", "fp8"]), "tol": rng.choice([3e-4, 1e-4, 1e-6]),
                "k_y": rng.choice([5, 10, 50])}
    if kind == "rank":
        pool = rng.choice([0, 0, 21])
        return {"kind": kind, "n": n // 21 * 21 if pool else n, "B": _log_int(rng, 1, 256),
                "K": rng.choice([10, 100, 1000]) if n >= 42000 else 10, "pool": pool}
    if kind == "observe":
        bf16 = rng.random() < 0.5
        d = 8 * _log_int(rng, 8, 256) if bf16 else _log_int(rng, 64, 512)
        n = n if bf16 else min(n, 51200000 // d)
        return {"kind": kind, "n": n, "d": d, "nq": _log_int(rng, 1, 256), "k_y": rng.choice([5, 10, 50]),
                "dtype": "bf16" if bf16 else "f32"}
    if kind == "graph":
        bf16 = rng.random() < 0.5
        n = _log_int(rng, 2000, 250000 if bf16 else 100000)
        d = 8 * _log_int(rng, 8, 64) if bf16 else _log_int(rng, 64, 512)
        return {"kind": kind, "n": n, "d": d, "k": rng.choice([10, 30, 50]), "dtype": "bf16" if bf16 else "f32"}
    if kind == "serve":
        slots = _log_int(rng, 4, 128)
        r = min(rng.choice([0, 50, 100, 200]), n // 20)
        return {"kind": kind, "n": n, "slots": slots, "requests": 2 * slots, "r": r,
                "storage": rng.choice(["bf16", "bf16", "fp8"])}
    s = max(100, min(75000, int(n * rng.uniform(0.02, 0.2))))
    return {"kind": kind, "n": n, "B": _log_int(rng, 1, 64), "s": s, "iters": 20, "k_y": rng.choice([5, 10])}


# ---------------------------------------------------------------- inputs
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFF)
    return g


def _clusters(case):
    """Items per cluster: 5,000 on the million-node database (200 clusters), fewer on smaller ones."""
    return max(20, min(5000, case["n"] // max(1, min(200, case["n"] // 40))))


def _affinity(case, seed):
    """A clustered k-NN-like graph with the degree and weights of the k = 50 graphs: every node picks
    HALF_DEGREE neighbours, P_IN of them in its own cluster and the rest anywhere, weights s^3.
    Ids carry no locality, as in a database stored in the order it was collected.
    Returns (row_ptr, col, val, members): members[c * size:(c + 1) * size] are cluster c's nodes."""
    n, size = case["n"], _clusters(case)
    g = _gen(seed, 1)
    members = torch.randperm(n, generator=g, device="cuda")
    place = torch.empty_like(members)
    place[members] = torch.arange(n, device="cuda")
    m = min(HALF_DEGREE, size - 1)
    u = torch.rand((n, m), generator=g, device="cuda")
    base = (place // size * size)[:, None]
    width = torch.clamp(n - base, max=size)
    inside = members[base + (torch.rand((n, m), generator=g, device="cuda", dtype=torch.float64) * width).long()]
    outside = torch.randint(0, n, (n, m), generator=g, device="cuda")
    dst = torch.where(u < P_IN, inside, outside)
    del inside, outside, u
    src = torch.arange(n, device="cuda")[:, None].expand(n, m)
    keep = (src != dst).reshape(-1)
    key = (torch.minimum(src, dst) * n + torch.maximum(src, dst)).reshape(-1)[keep]
    key = torch.unique(key)
    a, b = key // n, key % n
    w = (0.05 + 0.25 * torch.rand(key.numel(), generator=g, device="cuda")) ** 3
    both, order = torch.sort(torch.cat([key, b * n + a]))
    col = (both % n).int()
    val = torch.cat([w, w])[order]
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(both // n, minlength=n), 0)
    return row_ptr.int(), col, val, members


def _eigenpairs(case, rp, col, val, members, seed):
    """Approximate leading eigenpairs as a few Lanczos restarts leave them: an orthonormal basis of the
    D^1/2-weighted cluster indicators with sqrt(d) (eigenvalue 1) first."""
    n, r, size = case["n"], case["r"], _clusters(case)
    deg = torch.zeros(n, device="cuda", dtype=torch.float64)
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
    deg.index_add_(0, rows, val.double())
    del rows
    place = torch.empty_like(members)
    place[members] = torch.arange(n, device="cuda")
    label = torch.clamp(place // size, max=max(1, n // size) - 1)
    nc = int(label.max()) + 1
    if r > nc:  # more eigenpairs than clusters: halves, quarters, ... of them
        part = -(-r // nc)
        label = label * part + place % part
        nc = nc * part
    norm = torch.zeros(nc, device="cuda", dtype=torch.float64).index_add_(0, label, deg).sqrt()
    m = torch.randn((nc, r), generator=_gen(seed, 2), device="cuda", dtype=torch.float64)
    m[:, 0] = norm
    q = torch.linalg.qr(m)[0]
    u = (q[label] * (deg.sqrt() / torch.clamp(norm, min=1e-30)[label])[:, None]).float()
    lam = P_IN * np.linspace(1.0, 0.6, r)
    lam[0] = 1.0
    return lam, u.contiguous()


def _query_clusters(case, count, seed):
    """The cluster each query belongs to."""
    return np.random.default_rng([int(seed), 8]).integers(0, max(1, case["n"] // _clusters(case)), count)


def _observations(case, members, count, seed):
    """Sparse observations: k_y items of one cluster (some from elsewhere), values s^3, ids ascending."""
    n, size, k_y = case["n"], _clusters(case), case.get("k_y", 10)
    rng = np.random.default_rng([int(seed), 3, n])
    host = members.cpu().numpy()
    ptr, idx, val = [0], [], []
    for c in _query_clusters(case, count, seed):
        own = host[c * size + rng.choice(size, min(k_y, size), replace=False)]
        far = rng.integers(0, n, k_y)
        ids = np.unique(np.where(rng.random(own.size) < 0.8, own, far[:own.size]))
        idx.append(ids)
        val.append(rng.uniform(0.05, 0.3, ids.size) ** 3)
        ptr.append(ptr[-1] + ids.size)
    return np.asarray(ptr, np.int32), np.concatenate(idx).astype(np.int32), np.concatenate(val).astype(np.float32)


def _descriptors(rows, d, means, w, g):
    """Unit vectors around mixture means with mean cosine w, in blocks."""
    out = torch.empty((rows, d), device="cuda")
    for s in range(0, rows, 65536):
        e = min(rows, s + 65536)
        mu = means[torch.randint(0, means.shape[0], (e - s,), generator=g, device="cuda")]
        v = torch.randn((e - s, d), generator=g, device="cuda")
        v -= (v * mu).sum(1, keepdim=True) * mu
        v *= math.sqrt(1 - w * w) / v.norm(dim=1, keepdim=True)
        out[s:e] = v + w * mu
    return out


def _database(case, seed, nq):
    n, d = case["n"], case["d"]
    g = _gen(seed, 4)
    means = torch.randn((max(8, n // 100), d), generator=g, device="cuda")
    means /= means.norm(dim=1, keepdim=True)
    w = 2 * 50.0 / (d - 1 + math.sqrt((d - 1) ** 2 + 4 * 50.0 ** 2))  # mean cosine of a vMF sample, kappa = 50
    t = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    x = _descriptors(n, d, means, w, g).to(t)
    return x, _descriptors(nq, d, means, w, g).to(t) if nq else None


def _requests(case, members, seed):
    yp, yi, yv = _observations(case, members, case["requests"], seed)
    rng = np.random.default_rng([int(seed), 5])
    tol = rng.permutation(np.resize([1e-2, 1e-4, 1e-6], case["requests"]))
    top = rng.permutation(np.resize([10, 100, 1000] if case["n"] >= 4000 else [10, 100], case["requests"]))
    return [(yi[yp[j]:yp[j + 1]], yv[yp[j]:yp[j + 1]], float(tol[j]), int(top[j])) for j in range(case["requests"])]


def _shortlists(case, members, seed):
    """Per query the items of its own and the nearest clusters, in order of similarity (no order in their
    ids); lengths within a tenth of s, the first one exactly s."""
    n, s, B = case["n"], case["s"], case["B"]
    rng = np.random.default_rng([int(seed), 6, n])
    ptr, parts = [0], []
    for j, c in enumerate(_query_clusters(case, B, seed)):
        m = s if j == 0 else int(s * rng.uniform(0.9, 1.0))
        ids = members[(int(c) * _clusters(case) + torch.arange(m, device="cuda")) % n]
        parts.append(ids[torch.randperm(m, generator=_gen(seed, 100 + j), device="cuda")])
        ptr.append(ptr[-1] + m)
    return np.asarray(ptr, np.int32), torch.cat(parts).int()


def prepare(case, seed):
    kind = case["kind"]
    ctx = hd.Context(torch.cuda.current_device())
    st = {"kind": kind, "case": case, "ctx": ctx}
    if kind == "rank":
        g = _gen(seed, 7)
        # diffusion scores: positive and heavy-tailed
        st["x"] = torch.exp(2.0 * torch.randn((case["n"], case["B"]), generator=g, device="cuda"))
    elif kind in ("observe", "graph"):
        st["x"], st["q"] = _database(case, seed, case.get("nq", 0))
        if kind == "graph":  # room for the exported edges, at most 2 k a node
            st["col"] = np.zeros(2 * case["n"] * case["k"], np.int32)
            st["val"] = np.zeros(2 * case["n"] * case["k"], np.float32)
    else:
        rp, col, val, members = _affinity(case, seed)
        st["g"] = hd.graph_from_csr(ctx, rp, col, val)
        st["eig"] = None
        if case.get("r", 0) > 0:
            lam, u = _eigenpairs(case, rp, col, val, members, seed)
            st["eig"] = hd.eig_from_host(ctx, st["g"], lam, u, case["storage"])
        if kind == "serve":
            st["requests"] = _requests(case, members, seed)
            st["server"] = hd.Server(ctx, st["g"], st["eig"], "pcg" if st["eig"] else "paper", ALPHA,
                                     max_slots=case["slots"])
        else:
            st["y"] = _observations(case, members, case["B"], seed)
            if kind == "truncated":
                st["sl"] = _shortlists(case, members, seed)
                st["X"] = torch.empty((case["s"], case["B"]), device="cuda")
            else:
                st["X"] = torch.empty((case["n"], case["B"]), device="cuda")
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------- one pass
def run(st):
    kind, ctx, case = st["kind"], st["ctx"], st["case"]
    # the reported residual norms are left out everywhere: at these tolerances they measure what rounding leaves
    if kind == "query":
        x, it, _, status = hd.query_batch(ctx, st["g"], st["eig"], "pcg" if st["eig"] else "paper", *st["y"], ALPHA,
                                          case["tol"], 1000, X=st["X"])
        return {"x": x, "iters": it, "status": status}
    if kind == "rank":
        ids, score = hd.rank(ctx, st["x"], case["K"], pool=case["pool"])
        return {"ids": ids, "score": score}
    if kind == "observe":
        ptr, idx, val = hd.observe(ctx, st["x"], st["q"], case["k_y"], GAMMA)
        return {"ptr": ptr, "idx": idx, "val": val}
    if kind == "graph":
        rp, col, val, dinv = hd.build_graph(ctx, st["x"], case["k"], GAMMA).export()
        st["col"][:col.size] = col
        st["val"][:val.size] = val
        return {"row_ptr": rp, "col": st["col"], "val": st["val"], "dinv": dinv}
    if kind == "truncated":
        x, it, _, status = hd.temporal_truncated(ctx, st["g"], *st["sl"], *st["y"], ALPHA, 1e-12, case["iters"],
                                                 X=st["X"])
        return {"x": x, "iters": it, "status": status}
    server = st["server"]
    tickets = [server.submit(idx, val, tol, top) for idx, val, tol, top in st["requests"]]
    while server.step(1):
        pass
    server.completed(len(tickets))
    done = [server.poll(t, r[3]) for t, r in zip(tickets, st["requests"])]
    return {"ids": np.concatenate([d[0] for d in done]), "score": np.concatenate([d[1] for d in done]),
            "iters": np.asarray([d[2]["iters"] for d in done]), "status": np.asarray([d[2]["status"] for d in done])}


# ---------------------------------------------------------------- the bytes and operations of a pass
def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "rank":
        m = n * case["B"]
        return {"bytes": 4.0 * m + 8.0 * case["B"] * case["K"], "flops": float(m)}
    size = 2.0 if case.get("dtype") == "bf16" else 4.0
    if kind == "observe":
        return {"bytes": size * case["d"] * (n + case["nq"]) + 8.0 * case["nq"] * case["k_y"],
                "flops": 2.0 * n * case["nq"] * case["d"]}
    if kind == "graph":
        return {"bytes": size * case["d"] * n + 8.0 * n * 1.6 * case["k"], "flops": float(n) * n * case["d"]}
    nnz = 2.0 * HALF_DEGREE * n
    if kind == "truncated":
        rows = float(case["s"]) * case["B"]
        kept = 2.0 * HALF_DEGREE * P_IN * rows
        return {"bytes": 8.0 * nnz + 8.0 * rows, "flops": case["iters"] * (2.0 * kept + 10.0 * rows)}
    r, it = case["r"], 5 if case["r"] else 8
    u = n * r * {"f32": 4.0, "bf16": 2.0, "fp8": 1.0}[case["storage"]]
    B = case["B"] if kind == "query" else case["requests"]
    out = 4.0 * n * B if kind == "query" else 8.0 * 370 * B
    return {"bytes": 8.0 * nnz + 4.0 * n + u + out, "flops": it * B * (2.0 * nnz + 4.0 * n * r + 10.0 * n)}


# ---------------------------------------------------------------- the same in 64 bits
def _normalised(case, seed):
    rp, col, val, members = _affinity(case, seed)
    n = case["n"]
    deg = torch.zeros(n, device="cuda", dtype=torch.float64)
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
    deg.index_add_(0, rows, val.double())
    dinv = torch.where(deg > 0, deg.rsqrt(), torch.zeros_like(deg))
    w = val.double() * dinv[rows] * dinv[col.long()]
    return torch.sparse_csr_tensor(rp.long(), col.long(), w, size=(n, n), check_invariants=False), members, rows, val


def _solve(w, y, iters=None):
    """Columns of (I - a W) x = (1 - a) y by conjugate gradient: `iters` steps, or until 1e-13."""
    x, r = torch.zeros_like(y), y.clone()
    p, rr = r.clone(), (r * r).sum(0)
    first = rr.clone()
    for _ in range(iters or 400):
        q = (p - ALPHA * (w @ p)) / (1 - ALPHA)
        a = rr / torch.clamp((p * q).sum(0), min=1e-300)
        x += a * p
        r -= a * q
        new = (r * r).sum(0)
        if iters is None and bool((new <= 1e-26 * first).all()):
            break
        p = r + new / torch.clamp(rr, min=1e-300) * p
        rr = new
    return x


def _dense(n, yp, yi, yv, lo, hi):
    y = torch.zeros((n, hi - lo), device="cuda", dtype=torch.float64)
    for j in range(lo, hi):
        y[torch.from_numpy(yi[yp[j]:yp[j + 1]]).long().cuda(), j - lo] = torch.from_numpy(yv[yp[j]:yp[j + 1]]).double().cuda()
    return y


def _neighbours(x, q, k, exclude_self):
    """k largest inner products of each row of q with the rows of x (fp64)."""
    x64 = x.double() if x.numel() <= 1 << 28 else None
    best, ids = [], []
    for s in range(0, q.shape[0], 512):
        part = q[s:s + 512].double()
        if x64 is not None:
            sim = part @ x64.T
        else:
            sim = torch.cat([part @ c.double().T for c in x.split(1 << 16)], 1)
        if exclude_self:
            sim[torch.arange(part.shape[0]), torch.arange(s, s + part.shape[0])] = -math.inf
        top = torch.topk(sim, k, dim=1)
        best.append(top.values)
        ids.append(top.indices)
    return torch.cat(best), torch.cat(ids)


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "rank":
        x = prepare(case, seed)["x"].double()
        if case["pool"]:
            x = x.reshape(n // case["pool"], case["pool"], -1).sum(1)
        return {"ids": None, "score": torch.topk(x.T, case["K"], dim=1).values}
    if kind == "observe":
        x, q = _database(case, seed, case["nq"])
        sim, ids = _neighbours(x, q, case["k_y"], False)
        order = torch.argsort(ids, dim=1)
        val = torch.clamp(torch.gather(sim, 1, order), min=0) ** GAMMA
        return {"ptr": None, "idx": None, "val": val[val > 0]}
    if kind == "graph":
        if 2.0 * n * n * case["d"] > 1.1e13:
            return None  # the fp64 products alone would take more than ten seconds
        x, _ = _database(case, seed, 0)
        sim, ids = _neighbours(x, x, case["k"], True)
        w = (torch.clamp(sim, min=0) ** GAMMA).reshape(-1)
        i = torch.arange(n, device="cuda")[:, None].expand_as(ids).reshape(-1)
        j = ids.reshape(-1)
        key, inv = torch.unique(torch.minimum(i, j) * n + torch.maximum(i, j), return_inverse=True)
        edge = torch.zeros(key.numel(), device="cuda", dtype=torch.float64).scatter_reduce_(0, inv, w, "amax")
        deg = torch.zeros(n, device="cuda", dtype=torch.float64)
        deg.index_add_(0, key // n, edge).index_add_(0, key % n, edge)
        return {"row_ptr": None, "col": None, "val": None, "dinv": torch.where(deg > 0, deg.rsqrt(), 0 * deg)}
    w, members, rows, val = _normalised(case, seed)
    if kind == "query":
        yp, yi, yv = _observations(case, members, case["B"], seed)
        x = torch.empty((n, case["B"]), device="cuda", dtype=torch.float64)
        for lo in range(0, case["B"], 64):
            hi = min(case["B"], lo + 64)
            x[:, lo:hi] = _solve(w, _dense(n, yp, yi, yv, lo, hi))
        return {"x": x, "iters": None, "status": None}
    if kind == "serve":
        req = _requests(case, members, seed)
        score = []
        for lo in range(0, len(req), 64):
            part = req[lo:lo + 64]
            yp = np.concatenate([[0], np.cumsum([r[0].size for r in part])])
            x = _solve(w, _dense(n, yp, np.concatenate([r[0] for r in part]), np.concatenate([r[1] for r in part]),
                                 0, len(part)))
            score += [torch.topk(x[:, j], r[3]).values for j, r in enumerate(part)]
        return {"ids": None, "score": torch.cat(score), "iters": None, "status": None}
    yp, yi, yv = _observations(case, members, case["B"], seed)
    sp, si = _shortlists(case, members, seed)
    col = w.col_indices()
    x = torch.zeros((case["s"], case["B"]), device="cuda", dtype=torch.float64)
    for j in range(case["B"]):
        own = si[int(sp[j]):int(sp[j + 1])].long()
        pos = torch.full((n,), -1, device="cuda", dtype=torch.int64)
        pos[own] = torch.arange(own.numel(), device="cuda")
        keep = (pos[rows] >= 0) & (pos[col] >= 0)
        a, b, v = pos[rows[keep]], pos[col[keep]], val[keep].double()
        deg = torch.zeros(own.numel(), device="cuda", dtype=torch.float64).index_add_(0, a, v)
        dinv = torch.where(deg > 0, deg.rsqrt(), torch.zeros_like(deg))
        sub = torch.sparse_coo_tensor(torch.stack([a, b]), v * dinv[a] * dinv[b], (own.numel(),) * 2).to_sparse_csr()
        y = _dense(n, yp, yi, yv, j, j + 1)[own]
        x[:own.numel(), j:j + 1] = _solve(sub, y, case["iters"])
    return {"x": x, "iters": None, "status": None}

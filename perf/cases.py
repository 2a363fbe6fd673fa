"""What this library's speed is measured on: calls of its public entry points as a user's program makes them.

listed() holds the named cases, draw() further ones of the same ranges. Graphs are seeded R-MAT graphs (web and
social shape, (a, b, c, d) = (.57, .19, .19, .05)) and dropped-edge grids (road shape), the two families of the
benchmark; batches are 80 % uniform insertions and 20 % deletions of existing edges, or insertion-only stream
windows. Everything is generated on the GPU from the seed.

A pass (run) is one call, or the few calls one step of a program makes:
  static   Static PageRank of a resident graph, from 1/n or from given ranks (Naive-dynamic)
  dfp, dt  ranks after a batch that the graph already holds: DF-P (or DF), Dynamic Traversal
  update   a sliding window: a batch is applied and DF-P run, then the same edges leave again and DF-P runs again
  build    edge list in HBM -> graph handle, both CSRs read back
  ppr      K teleport columns on a weighted graph
  train    forward and backward of the K-column solve through autograd
"""
import math

import torch

import paper_2404_08299_gb300 as prdf

ALPHA, TOL, TAU, MAX_ITER = 0.85, 1e-10, 1e-6, 500
ABC = (0.57, 0.19, 0.19)


def listed():
    return [
        # the headline solve: ranks of a 16.8 M-vertex web-shaped graph from scratch
        {"name": "static-rmat24", "kind": "static", "graph": "rmat", "n": 1 << 24, "edges": 1 << 28, "precision": 0,
         "warm": False},
        # a small graph that fits L2: latency and launches count
        {"name": "static-rmat16", "kind": "static", "graph": "rmat", "n": 1 << 16, "edges": 1 << 20, "precision": 0,
         "warm": False},
        # road-shaped graph: every row short
        {"name": "static-grid4096", "kind": "static", "graph": "grid", "n": 4096 * 4096, "edges": 4 * 4096 * 4096,
         "precision": 0, "warm": False},
        # the mixed-precision option (FP32 sweeps, then FP64)
        {"name": "mixed-rmat22", "kind": "static", "graph": "rmat", "n": 1 << 22, "edges": 1 << 26, "precision": 1,
         "warm": False},
        # ranks after a batch of 1e-4 |E| on the large graph
        {"name": "dfp-rmat24", "kind": "dfp", "graph": "rmat", "n": 1 << 24, "edges": 1 << 28, "precision": 0,
         "fraction": 1e-4, "ins_only": False, "prune": 1},
        # a temporal stream on a 2^20-vertex graph: small insertion windows, apply and DF-P each
        {"name": "update-stream20", "kind": "update", "graph": "rmat", "n": 1 << 20, "edges": 15 << 20,
         "fraction": 1e-5, "ins_only": True},
        # Dynamic Traversal, odd sizes
        {"name": "dt-rmat22", "kind": "dt", "graph": "rmat", "n": 3000017, "edges": 50000003, "precision": 0,
         "fraction": 1e-5, "ins_only": False},
        # graph construction from an edge list, the first step of every program
        {"name": "build-rmat24", "kind": "build", "graph": "rmat", "n": 1 << 24, "edges": 1 << 28, "weighted": False},
        # the same with edge weights, what the K-column calls start from
        {"name": "build-weighted-rmat22", "kind": "build", "graph": "rmat", "n": 1 << 22, "edges": 1 << 26,
         "weighted": True},
        # 64 personalised columns at once, mixed precision
        {"name": "ppr-k64-rmat22", "kind": "ppr", "graph": "rmat", "n": 1 << 22, "edges": 1 << 26, "K": 64,
         "precision": 1},
        # few columns, ragged, FP64, on a small graph
        {"name": "ppr-k5-rmat16", "kind": "ppr", "graph": "rmat", "n": 50021, "edges": 700001, "K": 5,
         "precision": 0},
        # a learning step: gradients of the teleports and of the edge weights
        {"name": "train-k32-rmat19", "kind": "train", "graph": "rmat", "n": 1 << 19, "edges": 1 << 23, "K": 32,
         "precision": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["static", "static", "dfp", "dfp", "update", "dt", "build", "ppr", "train"])
    case = {"kind": kind, "graph": "rmat"}
    top = {"static": 1 << 24, "dfp": 1 << 24, "update": 1 << 22, "dt": 1 << 23, "build": 1 << 24, "ppr": 1 << 21,
           "train": 1 << 19}[kind]
    n = _log(rng, 1 << 13, top)
    if kind in ("static", "dfp") and rng.random() < 0.25:
        side = max(64, int(math.isqrt(n)))
        case.update(graph="grid", n=side * side, edges=4 * side * side)
    else:
        case.update(n=n, edges=int(n * rng.uniform(4, 16)))
    if kind == "static":
        case.update(precision=rng.choice([0, 0, 1]), warm=rng.random() < 0.3)
    elif kind in ("dfp", "dt"):
        case.update(precision=0, fraction=10 ** rng.uniform(-6, -2.5), ins_only=rng.random() < 0.3)
        if kind == "dfp":
            case.update(precision=rng.choice([0, 0, 0, 1]), prune=rng.choice([1, 1, 1, 0]))
    elif kind == "update":
        case.update(fraction=10 ** rng.uniform(-6, -4), ins_only=rng.random() < 0.5)
    elif kind == "build":
        case.update(weighted=rng.random() < 0.4)
        if case["weighted"]:
            case.update(n=min(case["n"], 1 << 22), edges=min(case["edges"], 1 << 26))
    else:
        case.update(K=rng.choice([1, 3, 5, 8, 16, 24, 33, 64]), precision=rng.choice([0, 1]) if kind == "ppr" else 1)
        if kind == "ppr" and case["precision"] == 0:  # FP64 steps cost three times the mixed solve's
            case.update(n=min(case["n"], 1 << 19), edges=min(case["edges"], 1 << 23))
    return case


# ---------------------------------------------------------------- inputs ----

def _rmat(n, edges, gen):
    """Raw R-MAT samples (duplicates and u == v included); ids beyond n fold back into [0, n)."""
    scale = max(1, (n - 1).bit_length())
    src = torch.empty(edges, dtype=torch.int32, device="cuda")
    dst = torch.empty(edges, dtype=torch.int32, device="cuda")
    a, b, c = ABC
    step = 1 << 25
    for i in range(0, edges, step):
        k = min(step, edges - i)
        u = torch.zeros(k, dtype=torch.int32, device="cuda")
        v = torch.zeros(k, dtype=torch.int32, device="cuda")
        for _ in range(scale):
            r = torch.rand(k, device="cuda", generator=gen)
            sb = r >= a + b
            db = ((r >= a) & ~sb) | (r >= a + b + c)
            u.mul_(2).add_(sb)
            v.mul_(2).add_(db)
        src[i:i + k] = u % n
        dst[i:i + k] = v % n
    return src, dst


def _grid(n, gen):
    """side x side 4-neighbour grid, both directions, each directed edge dropped with probability 0.05."""
    side = math.isqrt(n)
    ids = torch.arange(n, dtype=torch.int32, device="cuda").view(side, side)
    pairs = [(ids[1:], ids[:-1]), (ids[:-1], ids[1:]), (ids[:, 1:], ids[:, :-1]), (ids[:, :-1], ids[:, 1:])]
    src = torch.cat([p.reshape(-1) for p, _ in pairs])
    dst = torch.cat([q.reshape(-1) for _, q in pairs])
    keep = torch.rand(src.numel(), device="cuda", generator=gen) >= 0.05
    return src[keep].contiguous(), dst[keep].contiguous()


def _distinct(n, edges, gen):
    """`edges` distinct R-MAT edges without self-loops in random order, every twentieth given twice: where a pass
    returns one value an edge, their number is the same for every seed."""
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    while keys.numel() < edges:
        src, dst = _rmat(n, edges + edges // 4, gen)
        k = src.long() * n + dst.long()
        keys = torch.unique(torch.cat([keys, k[src != dst]]))
    keys = keys[torch.randperm(keys.numel(), device="cuda", generator=gen)[:edges]]
    keys = torch.cat([keys, keys[::20]])
    return (keys // n).int(), (keys % n).int()


def _edges(case, gen):
    if case["kind"] in ("build", "train"):
        return _distinct(case["n"], case["edges"], gen)
    return _grid(case["n"], gen) if case["graph"] == "grid" else _rmat(case["n"], case["edges"], gen)


def _batch(case, src, dst, gen):
    """(del_src, del_dst, ins_src, ins_dst): existing non-self-loop edges to delete and new pairs to insert, each
    once, so that applying the lists the other way round undoes the batch."""
    n, m = case["n"], src.numel()
    size = max(1, int(round(case["fraction"] * m)))
    n_del = 0 if case["ins_only"] else size // 5
    keys = torch.unique(src.long() * n + dst.long())
    pos = torch.randint(m, (2 * n_del + 8,), device="cuda", generator=gen)
    dk = torch.unique(src[pos].long() * n + dst[pos].long())
    dk = dk[dk // n != dk % n]
    dk = dk[torch.randperm(dk.numel(), device="cuda", generator=gen)][:n_del]
    ik = torch.unique(torch.randint(n * n, (2 * (size - n_del) + 8,), device="cuda", generator=gen))
    at = torch.searchsorted(keys, ik).clamp_(max=keys.numel() - 1)
    ik = ik[(keys[at] != ik) & (ik // n != ik % n)]
    ik = ik[torch.randperm(ik.numel(), device="cuda", generator=gen)][:size - n_del]
    return tuple(t.int().contiguous() for t in (dk // n, dk % n, ik // n, ik % n))


def _weights(m, gen):
    return 0.5 + torch.rand(m, device="cuda", generator=gen)


def _teleport(n, K, gen):
    """16 seed vertices a column with random weights that sum to 1."""
    S = torch.zeros(n, K, dtype=torch.float64, device="cuda")
    rows = torch.randint(n, (16, K), device="cuda", generator=gen)
    w = torch.rand(16, K, dtype=torch.float64, device="cuda", generator=gen) + 0.01
    S.scatter_add_(0, rows, w / w.sum(0))
    return S


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind, n = case["kind"], case["n"]
    src, dst = _edges(case, gen)
    st = {"case": case}
    if kind == "build":
        st.update(src=src, dst=dst, w=_weights(src.numel(), gen) if case["weighted"] else None)
        return st
    if kind in ("ppr", "train"):
        g = prdf.Graph(n, src, dst, _weights(src.numel(), gen))
        st.update(g=g, S=_teleport(n, case["K"], gen))
        if kind == "train":
            st["w"] = _weights(g.m, gen).requires_grad_()
            st["S"].requires_grad_()
            st["G"] = torch.randn(n, case["K"], dtype=torch.float64, device="cuda", generator=gen)
        return st
    g = prdf.Graph(n, src, dst)
    st["g"] = g
    if kind == "static":
        R0 = None
        if case["warm"]:
            R0 = torch.rand(n, dtype=torch.float64, device="cuda", generator=gen)
            R0 = R0 / R0.sum()
        st["R0"] = R0
        return st
    batch = _batch(case, src, dst, gen)
    st.update(batch=batch, prev=g.pagerank_static()[0])
    if kind != "update":
        st["masks"] = g.apply_batch(*batch)
    return st


# ------------------------------------------------------------------ pass ----

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "static":
        return state["g"].pagerank_static(R0=state["R0"], precision=case["precision"])[0]
    if kind in ("dfp", "dt"):
        ds, dd, is_, _ = state["batch"]
        de, ie = state["masks"]
        if kind == "dt":
            R, _, dV = state["g"].pagerank_dt(ds, dd, is_, state["prev"], del_mask=de, ins_mask=ie, want_dV=True)
            return [R, dV]
        if case["precision"]:  # the FP32 stage decides flags at FP32 resolution: ranks only
            return [state["g"].pagerank_dfp(ds, dd, is_, state["prev"], del_mask=de, ins_mask=ie,
                                            prune=case["prune"], precision=1)[0]]
        R, _, dV = state["g"].pagerank_dfp(ds, dd, is_, state["prev"], del_mask=de, ins_mask=ie, want_dV=True,
                                           prune=case["prune"])
        return [R, dV]
    if kind == "update":
        g = state["g"]
        ds, dd, is_, id_ = state["batch"]
        de, ie = g.apply_batch(ds, dd, is_, id_)
        R1, _, _ = g.pagerank_dfp(ds, dd, is_, state["prev"], del_mask=de, ins_mask=ie)
        ue, uf = g.apply_batch(is_, id_, ds, dd)
        R2, _, _ = g.pagerank_dfp(is_, id_, ds, R1, del_mask=ue, ins_mask=uf)
        return [de, ie, R1, ue, uf, R2]
    if kind == "build":
        g = prdf.Graph(case["n"], state["src"], state["dst"], state["w"])
        return [t for which in (prdf.PRDF_OUT, prdf.PRDF_IN) for t in g.export_csr(which) if t is not None]
    if kind == "ppr":
        return state["g"].pagerank_ppr(state["S"], precision=case["precision"])[0]
    R = prdf.PageRankFn.apply(state["g"], state["S"], state["w"], {"precision": case["precision"]})
    gS, gw = torch.autograd.grad(R, (state["S"], state["w"]), state["G"])
    return [R.detach(), gS, gw]


def work(case):
    """Compulsory bytes and operations of a pass. A solve streams the CSR (4 bytes an edge, 8 a vertex), the
    state and the result once per sweep; the number of sweeps to tolerance is a nominal one per kind."""
    n, m, K = case["n"], case["edges"] + case["n"], case.get("K", 1)
    kind = case["kind"]
    if kind == "build":  # edge list in; two CSRs out, each read back once
        w = 4 if case["weighted"] else 0
        return {"bytes": case["edges"] * (8 + w) + 2 * (m * (4 + w) + 8 * n), "flops": 0}
    if kind in ("ppr", "train"):
        sweeps = 70 * (2 if kind == "train" else 1)
        size = 8 if case["precision"] == 0 else 4
        return {"bytes": sweeps * (m * (4 + size) + 8 * n + 2 * size * n * K), "flops": 2 * sweeps * m * K}
    if kind in ("static", "dt"):
        sweeps = 40 if kind == "dt" or case["graph"] == "grid" else 60
        return {"bytes": sweeps * (4 * m + 24 * n), "flops": sweeps * m}
    # DF-P touches the affected part only: the ranks in and out, and a share of the graph that grows with the batch
    share = min(1.0, 4 * max(case["fraction"] * m, 1.0) ** 0.5 / n ** 0.5)
    per = share * 15 * (4 * m + 24 * n) + 16 * n
    if kind == "update":  # two batches merged into both CSRs (each copied once) and two DF-P calls
        return {"bytes": 2 * (per + 2 * (8 * m + 16 * n)), "flops": 2 * int(15 * share * m)}
    return {"bytes": per, "flops": int(15 * share * m)}


# ------------------------------------------------- the results in 64 bits ----

def _unique(n, src, dst, w=None):
    """Keys u * n + v of the edge set with one self-loop a vertex (w: the largest weight of equal edges, 1 on an
    added self-loop)."""
    loops = torch.arange(n, dtype=torch.int64, device="cuda")
    k = torch.cat([src.long() * n + dst.long(), loops * n + loops])
    if w is None:
        return torch.unique(k), None
    keys, at = torch.unique(k, return_inverse=True)
    ww = torch.cat([w.double(), torch.zeros(n, dtype=torch.float64, device="cuda")])
    out = torch.zeros(keys.numel(), dtype=torch.float64, device="cuda").scatter_reduce(0, at, ww, "amax")
    return keys, torch.where(out == 0, torch.ones_like(out), out)


def _pull(n, keys, val=None):
    """A with A[v, u] = val for the edge (u, v), in CSR form, and the out-degrees."""
    u, v = keys // n, keys % n
    deg = torch.bincount(u, minlength=n).double()
    t, at = torch.sort(v * n + u)
    rows = torch.searchsorted(t, torch.arange(n + 1, device="cuda") * n)
    val = torch.ones(keys.numel(), dtype=torch.float64, device="cuda") if val is None else val[at]
    return torch.sparse_csr_tensor(rows, t % n, val, size=(n, n)), deg


def _static(A, deg, n, R, dV=None):
    c0 = (1 - ALPHA) / n
    for _ in range(MAX_ITER):
        r = c0 + ALPHA * (A @ (R / deg))
        if dV is not None:
            r = torch.where(dV, r, R)
        done = float((r - R).abs().max()) <= TOL
        R = r
        if done:
            return R
    return R


def _mark(A, n, batch, masks):
    ds, dd, is_, _ = batch
    de, ie = (x.bool() for x in masks)
    dN = torch.zeros(n, dtype=torch.float64, device="cuda")
    dN[ds[de].long()] = 1
    dN[is_[ie].long()] = 1
    dV = torch.zeros(n, dtype=torch.bool, device="cuda")
    dV[dd[de].long()] = True
    return dV | ((A @ dN) > 0)


def _frontier(A, deg, n, R, dV, prune):
    c0 = (1 - ALPHA) / n
    for _ in range(MAX_ITER):
        x = R / deg
        c = A @ x
        r = (c0 + ALPHA * (c - x)) / (1 - ALPHA / deg) if prune else c0 + ALPHA * c
        r = torch.where(dV, r, R)
        dr, big = (r - R).abs(), torch.maximum(r, R)
        dN = dV & (dr > TAU * big)
        done = float(dr.max()) <= TOL
        if prune:
            dV = dV & ~(dr <= TAU * big)
        R = r
        if done:
            break
        dV = dV | ((A @ dN.double()) > 0)
    return R


def _columns(A, S, rhs):
    R = S.clone()
    for _ in range(MAX_ITER):
        r = ALPHA * (A @ R) + rhs
        done = float((r - R).abs().max()) <= 1e-13
        R = r
        if done:
            break
    return R


def _apply(keys, n, batch):
    ds, dd, is_, id_ = (x.long() for x in batch)
    keys = keys[~torch.isin(keys, ds * n + dd)]
    return torch.unique(torch.cat([keys, is_ * n + id_]))


def exact(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind, n = case["kind"], case["n"]
    src, dst = _edges(case, gen)
    uniform = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    if kind == "build":
        if not case["weighted"]:
            return None  # whole numbers only
        keys, w = _unique(n, src, dst, _weights(src.numel(), gen))
        return [None, None, w, None, None, w[torch.argsort(keys % n * n + keys // n)]]
    if kind in ("ppr", "train"):
        keys, w = _unique(n, src, dst, _weights(src.numel(), gen))
        S = _teleport(n, case["K"], gen)
        if kind == "train":
            w = _weights(keys.numel(), gen).double()
        u, v = keys // n, keys % n
        W = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, u, w)
        P = w / W[u]
        R = _columns(_pull(n, keys, P)[0], S, (1 - ALPHA) * S)
        if kind == "ppr":
            return R
        G = torch.randn(n, case["K"], dtype=torch.float64, device="cuda", generator=gen)
        off = torch.searchsorted(u, torch.arange(n + 1, device="cuda"))
        lam = _columns(torch.sparse_csr_tensor(off, v, P, size=(n, n)), G, G)
        own = (R * (lam - G)).sum(1)
        gw = torch.empty_like(w)
        for i in range(0, w.numel(), 1 << 22):
            s = slice(i, i + (1 << 22))
            gw[s] = (ALPHA * (R[u[s]] * lam[v[s]]).sum(1) - own[u[s]]) / W[u[s]]
        return [R, (1 - ALPHA) * lam, gw]
    keys = _unique(n, src, dst)[0]
    if kind == "static":
        A, deg = _pull(n, keys)
        R0 = uniform
        if case["warm"]:
            R0 = torch.rand(n, dtype=torch.float64, device="cuda", generator=gen)
            R0 = R0 / R0.sum()
        return _static(A, deg, n, R0)
    batch = _batch(case, src, dst, gen)
    del src, dst
    masks = [torch.ones(batch[i].numel(), dtype=torch.uint8, device="cuda") for i in (0, 2)]
    A, deg = _pull(n, keys)
    prev = _static(A, deg, n, uniform)
    after = _apply(keys, n, batch)
    A1, deg1 = _pull(n, after)
    dV = _mark(A1, n, batch, masks)
    if kind == "dt":
        new = dV
        while bool(new.any()):
            new = ((A1 @ new.double()) > 0) & ~dV
            dV = dV | new
        return [_static(A1, deg1, n, prev, dV), None]
    R1 = _frontier(A1, deg1, n, prev, dV, kind == "update" or case["prune"])
    if kind == "dfp":
        return [R1] if case["precision"] else [R1, None]
    undo = (batch[2], batch[3], batch[0], batch[1])
    R2 = _frontier(A, deg, n, R1, _mark(A, n, undo, masks[::-1]), True)
    return [None, None, R1, None, None, R2]

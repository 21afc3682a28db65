"""Performance cases: what a program asks of this package, through its public entry points.

Searches (FP32, BF16 and FP8 traversal; device and host buffers; one query to tens of thousands; uneven batches as a
captured plan), the exact kNN of the construction and of the ground truth, the pruning of Alg. 3, the reduced-precision
copies of the base rows, and a whole index build. Inputs follow the synthetic cross-modal recipe of ``roarsynth`` (unit
rows of Gaussian mixtures, queries shifted by one offset), drawn on the GPU. Searches walk a seeded navigable graph that
is made here from the inputs alone: in-component neighbours at spread ranks plus a few far links, about 30 ids of a 64-id
row as in a built index.
"""
import math

import numpy as np
import torch

import paper_2408_08933_gb300 as rg

BASE_N, BASE_D = 1_000_000, 200        # the base_1m_d200 workload
WIDE_D = 512                           # the base_1m_d512 workload
TINY_N, TINY_D = 10_000, 64            # the tiny workload
R = 64                                 # graph row width, 2M at M = 32
DEV = "cuda"
FORMS = ("f32", "bf16", "fp8")


def _search(form, nq, n, d, k, L, deleted=False, host=False):
    return {"op": "search", "form": form, "nq": nq, "n": n, "d": d, "k": k, "L": L, "deleted": deleted, "host": host}


def listed():
    return [
        # One interactive query against the 1M x 200 index: latency alone.
        dict(_search("f32", 1, BASE_N, BASE_D, 10, 100), name="search_f32_one"),
        # A request of a retrieval service, queries and answers in host memory, wide rows, top 100.
        dict(_search("bf16", 200, BASE_N, WIDE_D, 100, 200, host=True), name="search_bf16_request"),
        # The benchmark's batch: 10,000 test queries at recall@10 of 0.9.
        dict(_search("f32", 10_000, BASE_N, BASE_D, 10, 90), name="search_f32_batch"),
        # The smallest copy of the rows, with a tenth of them deleted.
        dict(_search("fp8", 10_000, BASE_N, BASE_D, 10, 100, deleted=True), name="search_fp8_batch"),
        # High recall on wide rows: long pools.
        dict(_search("bf16", 4_099, BASE_N, WIDE_D, 10, 350), name="search_bf16_long"),
        # Mixed k and L in one captured launch (the uneven benchmark).
        {"name": "uneven_bf16", "op": "uneven", "form": "bf16", "nq": 16_384, "n": BASE_N, "d": WIDE_D, "L": 500},
        # kNN of a small set, as a test or a notebook calls it.
        {"name": "knn_small", "op": "knn", "nt": 1_000, "n": TINY_N, "d": TINY_D, "kk": 50},
        # Ground truth of the test queries.
        {"name": "knn_truth", "op": "knn", "nt": 10_000, "n": BASE_N, "d": BASE_D, "kk": 10},
        # One block of training queries, the dense step of the construction.
        {"name": "knn_train", "op": "knn", "nt": 131_072, "n": BASE_N, "d": BASE_D, "kk": 100},
        # Pruning of one chunk of enhancement searches (pools of 500, some with reverse edges).
        {"name": "acquire_chunk", "op": "acquire", "nx": 65_536, "n": BASE_N, "d": BASE_D, "c": 532, "m": 32, "fill": False},
        # The reduced-precision copy a service makes of its base rows.
        {"name": "quantize_fp8", "op": "quantize", "form": "fp8", "n": BASE_N, "d": WIDE_D},
        # A whole construction at the tiny workload's size.
        {"name": "build_tiny", "op": "build", "n": TINY_N, "nt": TINY_N, "d": TINY_D, "depth": 100, "m": 32, "L": 100},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["search", "search", "search", "search", "uneven", "knn", "knn", "acquire", "quantize", "build"])
    n = _log(rng, 10_000, BASE_N)
    if op in ("search", "uneven"):
        form, d = rng.choice(FORMS), 4 * rng.randint(16, 128)
        if op == "uneven":
            return {"op": op, "form": form, "nq": _log(rng, 500, 16_384), "n": n, "d": d, "L": _log(rng, 100, 500)}
        k = rng.choice([1, 10, 10, 100, rng.randint(2, 99)])
        L = _log(rng, max(k, 10), 500)
        nq = _log(rng, 1, min(20_000, 20_000 * 100 * BASE_D // (L * d) + 1))
        return _search(form, nq, n, d, k, L, deleted=rng.random() < 0.2, host=rng.random() < 0.3)
    if op == "knn":
        d = 8 * rng.randint(8, 64)
        nt = _log(rng, 100, min(131_072, 131_072 * BASE_N * BASE_D // (n * d)))
        return {"op": op, "nt": nt, "n": n, "d": d, "kk": rng.choice([1, 10, 100, rng.randint(2, 99)])}
    if op == "acquire":
        d = 4 * rng.randint(16, 128)
        return {"op": op, "nx": _log(rng, 256, 65_536 * BASE_D // max(d, BASE_D)), "n": n, "d": d, "c": rng.randint(64, 532),
                "m": rng.choice([16, 32, 32, 35, 64]), "fill": rng.random() < 0.5}
    if op == "quantize":
        return {"op": op, "form": rng.choice(FORMS[1:]), "n": n, "d": 4 * rng.randint(16, 128)}
    n = _log(rng, 2_000, 20_000)
    return {"op": op, "n": n, "nt": _log(rng, n // 2, n), "d": 8 * rng.randint(8, 32), "depth": rng.randint(50, 100),
            "m": rng.choice([16, 32]), "L": rng.randint(64, 150)}


# ---- inputs -----------------------------------------------------------------------------------------------------------


def _comps(n):
    return max(4, int(math.sqrt(n) / 4))


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 7919 + 17)
    return g


def _unit(x):
    return x / x.norm(dim=1, keepdim=True)


def _rows(n, d, g, means, shift=None):
    comp = torch.randint(0, means.shape[0], (n,), generator=g, device=DEV)
    x = torch.randn(n, d, generator=g, device=DEV).mul_(0.5)
    x += means[comp]
    if shift is not None:
        x += shift
    x /= x.norm(dim=1, keepdim=True)
    return x, comp


def _inputs(n, d, nq, g):
    """Base rows with their components, and queries of the shifted mixture."""
    means = torch.randn(_comps(n), d, generator=g, device=DEV)
    X, comp = _rows(n, d, g, means)
    shift = 1.5 * _unit(torch.randn(1, d, generator=g, device=DEV))
    Q, _ = _rows(nq, d, g, means, shift)
    return X, comp, Q


def _blocks(X, comp):
    """Row ids by component, and for each component the similarities within it (its own diagonal below all)."""
    order = torch.argsort(comp, stable=True)
    ends = torch.cumsum(torch.bincount(comp, minlength=_comps(X.shape[0])), 0).tolist()
    lo = 0
    for hi in ends:
        if hi > lo:
            ids = order[lo:hi]
            Y = X[ids].to(torch.bfloat16)
            S = (Y @ Y.T).float()
            S.fill_diagonal_(-2.0)
            yield ids, S
        lo = hi


def _graph(X, comp, g):
    """A navigable graph, int32 [n, R]: neighbours of the own component at spread ranks, random members of it and far
    rows; no self links and no duplicates, padded with -1 at the end."""
    n = X.shape[0]
    near, spread, inside, far = 8, 12, 5, 7
    w = near + spread + inside + far
    adj = torch.full((n, w), -1, dtype=torch.int64, device=DEV)
    for ids, S in _blocks(X, comp):
        m = ids.shape[0]
        top = S.topk(min(m, 256), dim=1).indices
        K = top.shape[1]
        u = torch.rand(m, spread, generator=g, device=DEV)
        rank = (near * (K / near) ** u).long().clamp_(max=K - 1)
        pick = torch.randint(0, m, (m, inside), generator=g, device=DEV)
        adj[ids, :min(near, K)] = ids[top[:, :near]]
        adj[ids, near:near + spread] = ids[torch.gather(top, 1, rank)]
        adj[ids, near + spread:near + spread + inside] = ids[pick]
    adj[:, -far:] = torch.randint(0, n, (n, far), generator=g, device=DEV)
    adj[adj == torch.arange(n, device=DEV)[:, None]] = -1
    adj = adj.sort(dim=1, descending=True).values
    adj[:, 1:][adj[:, 1:] == adj[:, :-1]] = -1
    adj = adj.sort(dim=1, descending=True).values
    out = torch.full((n, R), -1, dtype=torch.int32, device=DEV)
    out[:, :w] = adj.int()
    return out


def _entry(X):
    """The row nearest to the mean of the rows."""
    return int((X - X.mean(dim=0, keepdim=True)).square().sum(dim=1).argmin())


def _copy(X, form):
    """The traversal copy of the rows and its scales."""
    if form == "f32":
        return None, None
    if form == "bf16":
        return X.to(torch.bfloat16).view(torch.int16), None
    s = X.abs().amax(dim=1) / 448.0
    s[s == 0] = 1.0
    return (X / s[:, None]).to(torch.float8_e4m3fn).view(torch.uint8), s


def _uneven_params(nq, L, g):
    """k of 1, 10 and 100 in equal shares, L uniform between max(k, 10) and the widest."""
    k = torch.tensor([1, 10, 100], device=DEV, dtype=torch.int32).repeat(nq // 3 + 1)[:nq]
    k = k[torch.randperm(nq, generator=g, device=DEV)]
    lo = k.clamp(min=10)
    Ls = lo + (torch.rand(nq, generator=g, device=DEV) * (L - lo + 1)).int()
    return k, Ls.clamp(max=L)


def _candidates(X, comp, nx, c, g):
    """Nodes and for each the nearest rows of its component (a final search pool) and a few others (reverse edges),
    at most c ids, int32 padded with -1, and their number."""
    n = X.shape[0]
    xs = torch.randperm(n, generator=g, device=DEV)[:min(nx, n)]
    if nx > n:
        xs = torch.cat([xs, torch.randint(0, n, (nx - n,), generator=g, device=DEV)])
    slot = torch.full((n,), -1, dtype=torch.int64, device=DEV)
    slot[xs] = torch.arange(nx, device=DEV)
    cand = torch.randint(0, n, (nx, c), generator=g, device=DEV)
    pool = c - c // 16
    for ids, S in _blocks(X, comp):
        at = slot[ids]
        mine = at >= 0
        K = min(ids.shape[0], pool)
        cand[at[mine], :K] = ids[S[mine].topk(K, dim=1).indices]
    count = pool + torch.randint(0, c - pool + 1, (nx,), generator=g, device=DEV)
    cand[torch.arange(c, device=DEV)[None, :] >= count[:, None]] = -1
    return xs.int(), cand.int(), count.int()


def _made(case, seed):
    """The plain inputs of a case: tensors and numbers, nothing of the package."""
    g, op = _gen(seed), case["op"]
    if op in ("search", "uneven"):
        X, comp, Q = _inputs(case["n"], case["d"], case["nq"], g)
        m = {"X": X, "Q": Q, "adj": _graph(X, comp, g), "entry": _entry(X), "tomb": None}
        m["trav"], m["scales"] = _copy(X, case["form"])
        if op == "uneven":
            m["k"], m["L"] = _uneven_params(case["nq"], case["L"], g)
        elif case["deleted"]:
            words = (case["n"] + 31) // 32
            dead = torch.rand(words, 32, generator=g, device=DEV) < 0.1
            m["tomb"] = (dead.long() << torch.arange(32, device=DEV)).sum(dim=1).to(torch.int32)
            m["dead"] = dead.reshape(-1)[:case["n"]]
        return m
    if op in ("knn", "build"):
        X, _, T = _inputs(case["n"], case["d"], case["nt"], g)
        return {"X": X, "T": T}
    X, comp, _ = _inputs(case["n"], case["d"], 1, g)
    if op == "acquire":
        xs, cand, count = _candidates(X, comp, case["nx"], case["c"], g)
        return {"X": X, "xs": xs, "cand": cand, "count": count}
    return {"X": X}


def prepare(case, seed):
    s = _made(case, seed)
    s["case"] = case
    if case["op"] in ("search", "uneven"):
        s["index"] = rg.Index(s["X"], s["adj"], s["entry"], dtype=case["form"], trav=s["trav"], scales=s["scales"])
        if s["tomb"] is not None:
            s["index"].set_tombstones(s["tomb"])
        if case["op"] == "uneven":
            s["out"] = s["index"].uneven_outputs(s["k"].cpu().numpy())
            s["plan"] = s["index"].plan_uneven(s["Q"], s["k"], s["L"], case["L"], s["out"])
        elif case["host"]:
            s["Q"] = s["Q"].cpu().pin_memory()
            k, nq = case["k"], case["nq"]
            s["out"] = tuple(torch.empty(shape, dtype=t, pin_memory=True) for shape, t in (
                ((nq, k), torch.int32), ((nq, k), torch.float32), (nq, torch.int32), (nq, torch.int32), (nq, torch.int32)))
    return s


def run(state):
    case, op = state["case"], state["case"]["op"]
    if op == "search":
        if case["host"]:
            return state["index"].search_host(state["Q"], case["k"], case["L"], out=state["out"])
        return state["index"].search(state["Q"], case["k"], case["L"])
    if op == "uneven":
        state["plan"].launch()
        return state["out"][1:]
    if op == "knn":
        return rg.knn(state["T"], state["X"], case["kk"])
    if op == "acquire":
        return rg.acquire(state["X"], state["xs"], state["cand"], state["count"], case["m"], case["fill"], sorted_out=True)
    if op == "quantize":
        codes, scales = rg.quantize(state["X"], case["form"])
        return codes if scales is None else (codes, scales)
    adj, entry, _ = rg.build_index(state["X"], state["T"], case["depth"], case["m"], case["L"])
    return adj, entry


# ---- the work of a pass -----------------------------------------------------------------------------------------------


def _visits(n, L):
    """Rows scored and nodes expanded by one query of beam width L (fitted to searches of these graphs)."""
    return min(0.8 * n, 150.0 * L ** 0.64), 1.04 * L + 18


def work(case):
    op = case["op"]
    if op in ("search", "uneven"):
        n, d, nq, b = case["n"], case["d"], case["nq"], {"f32": 4, "bf16": 2, "fp8": 1}[case["form"]]
        k = 37 if op == "uneven" else case["k"]
        L = (case["L"] + 37) / 2 if op == "uneven" else case["L"]
        v, h = _visits(n, L)
        low = b < 4
        row = d * b + (4 if b == 1 else 0)
        return {"bytes": nq * (v * row + h * 30 * 4 + (L * d * 4 if low else 0) + 4 * d + 8 * k + 12),
                "flops": 2.0 * nq * d * (v + (L if low else 0))}
    if op == "quantize":
        b = 2 if case["form"] == "bf16" else 1
        return {"bytes": case["n"] * (case["d"] * (4 + b) + (4 if b == 1 else 0)), "flops": case["n"] * case["d"]}
    if op == "acquire":
        nx, n, d, c, m = (case[i] for i in ("nx", "n", "d", "c", "m"))
        return {"bytes": 4 * (d * min(n, nx * c) + nx * (2 * c + m + 3)), "flops": 4.0 * nx * c * d}
    n, nt, d = case["n"], case["nt"], case["d"]
    if op == "knn":
        return {"bytes": 4 * d * (n + nt) + 8 * nt * case["kk"], "flops": 2.0 * n * nt * d}
    v, h = _visits(n, case["L"])
    return {"bytes": 4 * d * (n + nt) + n * (v * d * 4 + h * 30 * 4 + 8 * case["m"]),
            "flops": 2.0 * d * (n * nt + n * v + 2 * n * case["L"])}


# ---- the same in 64 bits ----------------------------------------------------------------------------------------------


def _decoded(m, form):
    if form == "f32":
        return m["X"]
    if form == "bf16":
        return m["trav"].view(torch.bfloat16).float()
    return m["trav"].view(torch.float8_e4m3fn).float()


def _beam(m, form, Q, L):
    """Beam search of width L[i] for every row of Q in 64 bits: the final pools (distance, id), sorted."""
    rows, adj, nq, n = _decoded(m, form), m["adj"].long(), Q.shape[0], m["X"].shape[0]
    Q, W, ar = Q.double(), int(L.max()), torch.arange(Q.shape[0], device=DEV)

    def dist(q, ids):
        d = -torch.einsum("qd,qjd->qj", q, rows[ids].double())
        return d * m["scales"][ids].double() if m["scales"] is not None else d

    inf = float("inf")
    pd = torch.full((nq, W), inf, dtype=torch.float64, device=DEV)
    pi = torch.zeros((nq, W), dtype=torch.int64, device=DEV)
    done = torch.ones((nq, W), dtype=torch.bool, device=DEV)
    inside = torch.arange(W, device=DEV)[None, :] < L[:, None]
    seen = torch.zeros((nq, n), dtype=torch.bool, device=DEV)
    start = torch.full((nq, 1), m["entry"], dtype=torch.int64, device=DEV)
    pd[:, :1], pi[:, :1] = dist(Q, start), start
    done[:, 0] = False
    seen[:, m["entry"]] = True
    while True:
        live = ar[~done.all(dim=1)]
        if live.numel() == 0:
            return pd, pi
        at = (~done[live]).int().argmax(dim=1)
        nb = adj[pi[live, at]]
        done[live, at] = True
        at = nb.clamp(min=0)
        fresh = (nb >= 0) & ~seen[live[:, None], at]
        seen[live[:, None].expand_as(at)[fresh], at[fresh]] = True
        d = dist(Q[live], at).masked_fill_(~fresh, inf)
        d, o = torch.cat([pd[live], d], dim=1).sort(dim=1, stable=True)
        i = torch.cat([pi[live], at], dim=1).gather(1, o)
        x = torch.cat([done[live], ~fresh], dim=1).gather(1, o)
        d, i, x = d[:, :W], i[:, :W], x[:, :W]
        out = ~inside[live]
        pd[live], pi[live], done[live] = d.masked_fill(out, inf), i, x | out


def _answers(m, form, Q, L):
    pd, pi = _beam(m, form, Q, L)
    if form != "f32":
        again = -torch.einsum("qd,qjd->qj", Q.double(), m["X"][pi].double())
        pd = again.masked_fill_(torch.isinf(pd), float("inf"))
    if m["tomb"] is not None:
        pd = pd.masked_fill(m["dead"][pi], float("inf"))
    return pd.sort(dim=1).values


def _blocks_of(total, size):
    return [slice(lo, min(total, lo + size)) for lo in range(0, total, size)]


def _exact_search(case, m):
    nq, n, d = case["nq"], case["n"], case["d"]
    uneven = case["op"] == "uneven"
    if nq * case["L"] * d * (0.5 if uneven else 1.0) > 4e9:
        return None
    L = m["L"].long() if uneven else torch.full((nq,), case["L"], dtype=torch.int64, device=DEV)
    got = []
    for b in _blocks_of(nq, max(1, min(2048, int(4e9 / n), int(1e9 / (R * d))))):
        d = _answers(m, case["form"], m["Q"][b], L[b])
        if uneven:
            ks = m["k"][b].long()
            d = d[torch.arange(d.shape[1], device=DEV)[None, :] < ks[:, None]]
        else:
            d = d[:, :case["k"]]
        got.append(d)
    got = torch.cat(got)
    return [None, got, None, None, None]


def _exact_knn(case, m):
    X, T, kk = m["X"], m["T"], case["kk"]
    got = []
    for b in _blocks_of(T.shape[0], max(1, int(1e9 / X.shape[0]))):
        S = T[b] @ X.T
        near = S.topk(min(kk + 16, X.shape[0]), dim=1).indices
        d = [-torch.einsum("qd,qjd->qj", T[b][c].double(), X[near[c]].double()) for c in _blocks_of(near.shape[0], 512)]
        got.append(torch.cat(d).sort(dim=1).values[:, :kk])
    return [None, torch.cat(got)]


def exact(case, seed):
    if case["op"] in ("acquire", "build"):
        return None                       # whole numbers only
    m = _made(case, seed)
    if case["op"] == "quantize":
        if case["form"] == "bf16":
            return None                   # codes only
        s = m["X"].abs().amax(dim=1).double() / 448.0
        return [None, torch.where(s == 0, torch.ones_like(s), s)]
    return _exact_knn(case, m) if case["op"] == "knn" else _exact_search(case, m)

"""The measured cases of this library: what its users have it do, through its public entry points.

A case names an entry point (``call``), an input family and its sizes; inputs are drawn on the GPU from
the seed alone.  The families are those of the library's own workloads (Barabasi-Albert, Erdos-Renyi,
random geometric, R-MAT 0.57/0.19/0.19/0.05, Chung-Lu 2.1) over the sizes those workloads use.

Calls:
  count        harp_count4 on a resident handle
  edges        count4_edges: build from an edge list (host arrays or device tensors), count, free
  batch        harp_batch_count on a prepared batch of many uneven graphs (captured CUDA graph)
  orbits       harp_count4_orbits, eleven roles per vertex, device output
  edge_orbits  harp_count4_edge_orbits, ten roles per edge, device output
  literal      harp_count4 under the literal basis
  serve        a burst of requests through the continuous-batching server, all results awaited
  partitioned  harp_count4_partitioned: host edge list, owner-rule blocks under a device budget
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_12074_gb300 import harp as H

DEV = "cuda"


# ---------------------------------------------------------------------------------------------
# Cases.
# ---------------------------------------------------------------------------------------------
def listed():
    return [
        # one small graph, handle kept: the latency of a single count (8 k edges, social skew)
        {"name": "count_ba_2k", "call": "count", "family": "ba", "n": 2000, "k": 8.0},
        # the same size from a host edge list: the smallest complete request of a user's script
        {"name": "edges_ba_2k_host", "call": "edges", "family": "ba", "n": 1999, "k": 8.0, "host": True},
        # the plain large skewed graph: R-MAT scale 20, edge factor 16, one graph per launch
        {"name": "count_rmat_20", "call": "count", "family": "rmat", "n": 1 << 20, "k": 32.0},
        # a large unskewed, localised graph (biological stand-in), odd vertex count
        {"name": "count_rgg_1m", "call": "count", "family": "rgg", "n": 1_000_003, "k": 16.0},
        # heavy-tailed web-like graph whose CSR exceeds L2 (the shape of the partitioned workload)
        {"name": "count_chung_lu_2m", "call": "count", "family": "chung_lu", "n": 2_000_000, "k": 48.0},
        # a complete request on a mid-size skewed graph already on the device: build, count, free
        {"name": "edges_rmat_18_device", "call": "edges", "family": "rmat", "n": 1 << 18, "k": 31.0, "host": False},
        # 4,096 graphs of uneven size in one captured launch
        {"name": "batch_4096", "call": "batch", "graphs": 4096, "n_lo": 50, "n_hi": 20000},
        # per-vertex roles of a mid-size skewed graph
        {"name": "orbits_rmat_15", "call": "orbits", "family": "rmat", "n": 1 << 15, "k": 32.0},
        # per-edge roles of a mid-size sparse graph with hubs
        {"name": "edge_orbits_ba_100k", "call": "edge_orbits", "family": "ba", "n": 100_001, "k": 12.0},
        # the equations as printed, on a small skewed graph
        {"name": "literal_rmat_13", "call": "literal", "family": "rmat", "n": 1 << 13, "k": 32.0},
        # a burst of mixed requests (edge counts log-uniform over the served range) through the server
        {"name": "serve_48", "call": "serve", "requests": 48, "m_lo": 1000, "m_hi": 10_000_000},
        # a host edge list counted in blocks under a device budget
        {"name": "partitioned_2m", "call": "partitioned", "family": "chung_lu", "n": 2_000_000, "k": 24.0,
         "budget_mb": 512},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sized(rng, family, m):
    """A graph of the family with about m edges: (n, mean degree)."""
    if family == "rmat":  # edge factors around 16 on a power-of-two vertex count
        n = 1 << max(6, int(round(math.log2(max(m, 1024) / 16.0))))
        return n, round(2.0 * m / n, 3)
    if family == "ba":
        a = rng.randint(2, 8)
        return max(a + 2, m // a), 2.0 * a
    k = round(rng.uniform(4.0, 32.0) if family != "chung_lu" else rng.uniform(8.0, 48.0), 3)
    return max(64, int(round(2 * m / k))), k


def draw(rng):
    call = rng.choice(["count", "count", "count", "edges", "edges", "batch", "orbits", "edge_orbits", "literal",
                       "serve", "partitioned"])
    if call == "batch":
        return {"call": call, "graphs": _log_uniform(rng, 16, 4096), "n_lo": 50, "n_hi": _log_uniform(rng, 2000, 20000)}
    if call == "serve":
        return {"call": call, "requests": _log_uniform(rng, 8, 48), "m_lo": 1000, "m_hi": _log_uniform(rng, 10**5, 10**7)}
    # families and edge counts each call is used with
    families, lo, hi = {
        "count": (["ba", "er", "rgg", "rmat", "chung_lu"], 3_000, 16_000_000),
        "edges": (["ba", "er", "rgg", "rmat"], 1_000, 10_000_000),
        "orbits": (["ba", "er", "rgg", "rmat"], 3_000, 500_000),
        "edge_orbits": (["ba", "er", "rgg", "rmat"], 3_000, 500_000),
        "literal": (["ba", "er", "rgg", "rmat"], 3_000, 130_000),
        "partitioned": (["ba", "rgg", "chung_lu"], 1_000_000, 24_000_000),
    }[call]
    family = rng.choice(families)
    n, k = _sized(rng, family, _log_uniform(rng, lo, hi))
    case = {"call": call, "family": family, "n": n, "k": k}
    if call == "edges":
        case["host"] = rng.random() < 0.5
    if call == "partitioned":
        # the triangle scratch (about 320 MB), a wedge block's per-vertex arrays, and part of the arcs
        case["budget_mb"] = int(320 + 105 * n / 1e6 + rng.uniform(4.0, 12.0) * n * k / 2e6)
    return case


# ---------------------------------------------------------------------------------------------
# Inputs: every generator draws many graphs at once.  ns, ks: python lists; returns local int32 src,
# dst on the device and each graph's edge bounds (python list of len(ns) + 1).
# ---------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1_000_003 + 17)
    return g


def _i64(values):
    return torch.tensor(values, dtype=torch.int64, device=DEV)


def _bounds(counts):
    out = [0]
    for c in counts:
        out.append(out[-1] + int(c))
    return out


def _owner(counts):
    """(graph of each item, index of the item within its graph) for counts items per graph."""
    c = _i64(counts)
    gid = torch.repeat_interleave(torch.arange(len(counts), device=DEV), c)
    start = torch.cumsum(c, 0) - c
    return gid, torch.arange(gid.numel(), device=DEV) - start[gid], start


def _er(ns, ks, gen):
    """Uniform pairs, n k / 2 of them (self-loops and repeats are dropped by the build)."""
    counts = [max(1, int(round(n * k / 2))) for n, k in zip(ns, ks)]
    gid, _, _ = _owner(counts)
    n = _i64(ns)[gid]
    pick = lambda: (torch.rand(gid.numel(), generator=gen, device=DEV, dtype=torch.float64) * n).long()  # noqa: E731
    return pick().int(), pick().int(), _bounds(counts)


def _ba(ns, ks, gen):
    """Preferential attachment, k / 2 edges per new vertex: edge e of a graph joins vertex 1 + e // a to a
    uniform earlier endpoint; endpoint slots that name another edge's target are resolved by following them."""
    a = [max(1, int(round(k / 2))) for k in ks]
    counts = [(n - 1) * d for n, d in zip(ns, a)]
    gid, e, start = _owner(counts)
    src = 1 + e // _i64(a)[gid]
    # slots 0 .. 2e of the endpoint list before edge e: slot 0 is vertex 0, slot 2j + 1 the source and
    # slot 2j + 2 the target of edge j
    slot = (torch.rand(gid.numel(), generator=gen, device=DEV, dtype=torch.float64) * (2 * e + 1)).long()
    base = start[gid]
    while True:
        follow = (slot > 0) & (slot % 2 == 0)
        if not bool(follow.any()):
            break
        j = torch.where(follow, slot // 2 - 1, torch.zeros_like(slot))
        slot = torch.where(follow, slot[base + j], slot)
    dst = torch.where(slot == 0, torch.zeros_like(slot), src[base + torch.clamp(slot // 2, min=0)])
    return src.int(), dst.int(), _bounds(counts)


def _rgg(ns, ks, gen):
    """Points in the unit square joined within the radius of mean degree k."""
    gid, _, start = _owner(ns)
    r = torch.tensor([math.sqrt(k / (math.pi * max(1, n - 1))) for n, k in zip(ns, ks)], dtype=torch.float64, device=DEV)
    side = torch.clamp((1.0 / r).floor().long(), min=1)
    cell0 = torch.cumsum(side * side, 0) - side * side
    x = torch.rand(gid.numel(), generator=gen, device=DEV, dtype=torch.float64)
    y = torch.rand(gid.numel(), generator=gen, device=DEV, dtype=torch.float64)
    s = side[gid]
    cx, cy = torch.minimum((x * s).long(), s - 1), torch.minimum((y * s).long(), s - 1)
    cell = cell0[gid] + cy * s + cx
    cell, order = torch.sort(cell)
    x, y, cx, cy, gid = x[order], y[order], cx[order], cy[order], gid[order]
    s, row0, local = side[gid], cell0[gid], order - start[gid]
    i = torch.arange(gid.numel(), device=DEV)
    us, vs = [], []
    for dy in (0, 1):  # the rest of this row's cells up to cx + 1, then the next row's cx - 1 .. cx + 1
        row = row0 + (cy + dy) * s
        right = row + torch.minimum(cx + 1, s - 1)
        hi = torch.searchsorted(cell, right, right=True)
        lo = i + 1 if dy == 0 else torch.searchsorted(cell, row + torch.clamp(cx - 1, min=0))
        c = torch.clamp(hi - lo, min=0)
        if dy == 1:
            c = torch.where(cy + 1 < s, c, torch.zeros_like(c))
        u = torch.repeat_interleave(i, c)
        v = torch.arange(u.numel(), device=DEV) - (torch.cumsum(c, 0) - c)[u] + lo[u]
        near = (x[u] - x[v]) ** 2 + (y[u] - y[v]) ** 2 <= r[gid[u]] ** 2
        us.append(u[near])
        vs.append(v[near])
    u, v = torch.cat(us), torch.cat(vs)
    eg, order = torch.sort(gid[u], stable=True)
    counts = torch.bincount(eg, minlength=len(ns)).tolist()
    return local[u][order].int(), local[v][order].int(), _bounds(counts)


def _rmat(n, k, gen):
    scale, m = n.bit_length() - 1, max(1, int(round(n * k / 2)))
    src = torch.zeros(m, dtype=torch.int64, device=DEV)
    dst = torch.zeros(m, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        p = torch.rand(m, generator=gen, device=DEV)
        src = 2 * src + (p >= 0.76).long()
        dst = 2 * dst + (((p >= 0.57) & (p < 0.76)) | (p >= 0.95)).long()
    perm = torch.randperm(n, generator=gen, device=DEV)
    return perm[src].int(), perm[dst].int()


def _chung_lu(n, k, gen):
    """n k / 2 pairs of endpoints drawn by weight (i + i0)^(-1/1.1), the largest expected degree n / 50."""
    ex, top = -1.0 / 1.1, max(4.0, n / 50.0)
    lo, hi = 1e-6, float(n)
    for _ in range(100):  # total weight n k with the first weight at top
        i0 = math.sqrt(lo * hi)
        c = top * i0 ** -ex
        total = c * (((n - 1 + i0) ** (ex + 1) - i0 ** (ex + 1)) / (ex + 1) + i0 ** ex)
        lo, hi = (lo, i0) if total > n * k else (i0, hi)
    w = (torch.arange(n, dtype=torch.float64, device=DEV) + i0) ** ex
    cum = torch.cumsum(w, 0)
    m = max(1, int(round(n * k / 2)))
    pick = lambda: torch.clamp(torch.searchsorted(  # noqa: E731
        cum, torch.rand(m, generator=gen, device=DEV, dtype=torch.float64) * cum[-1]), max=n - 1)
    return pick().int(), pick().int()


def _graph(family, n, k, seed):
    gen = _gen(seed)
    if family == "rmat":
        return _rmat(n, k, gen)
    if family == "chung_lu":
        return _chung_lu(n, k, gen)
    src, dst, _ = {"er": _er, "ba": _ba, "rgg": _rgg}[family]([n], [k], gen)
    return src, dst


def _spread(i, step):
    """A fixed low-discrepancy number in [0, 1) (so a case's sizes are the same for every seed)."""
    return (0.5 + i * step) % 1.0


def _members(case):
    """(family, n, k) of each member of a batch or of a burst: families in turn, sizes log-uniform."""
    out = []
    if case["call"] == "batch":
        for i in range(case["graphs"]):
            family = ("er", "ba", "rgg")[i % 3]
            u = (i // 3 + 0.5) / math.ceil(case["graphs"] / 3)
            n = int(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** u))
            v = _spread(i, 0.6180339887498949)
            out.append((family, n, 2.0 * (2 + int(7 * v)) if family == "ba" else 4.0 + 28.0 * v))
        return out
    for i in range(case["requests"]):
        family = ("er", "ba", "rgg", "rmat")[i % 4]
        u = (i + 0.5) / case["requests"]
        m = case["m_lo"] * (case["m_hi"] / case["m_lo"]) ** u
        v = _spread(i, 0.6180339887498949)
        if family == "rmat":
            n = 1 << max(4, int(round(math.log2(max(m, 16) / 16))))
            out.append((family, n, 32.0))
            continue
        k = 2.0 * (2 + int(7 * v)) if family == "ba" else 4.0 + 28.0 * v
        out.append((family, max(16, int(round(2 * m / k))), k))
    return out


def _member_edges(members, seed):
    """[(n, src, dst)] on the device, in the members' order."""
    out = [None] * len(members)
    for f, (family, make) in enumerate((("er", _er), ("ba", _ba), ("rgg", _rgg))):
        idx = [i for i, mem in enumerate(members) if mem[0] == family]
        if not idx:
            continue
        src, dst, at = make([members[i][1] for i in idx], [members[i][2] for i in idx], _gen(8 * seed + f))
        for j, i in enumerate(idx):
            out[i] = (members[i][1], src[at[j]:at[j + 1]], dst[at[j]:at[j + 1]])
    for i, (family, n, k) in enumerate(members):
        if family == "rmat":
            out[i] = (n, *_rmat(n, k, _gen(8 * seed + 7 + 4096 * i)))
    return out


def prepare(case, seed):
    call = case["call"]
    if call == "batch":
        graphs = [H.harp_build_csr(n, src, dst) for n, src, dst in _member_edges(_members(case), seed)]
        batch = H.harp_batch_create(graphs)  # the batch holds its own copy of the members
        for g in graphs:
            g.close()
        return {"call": call, "batch": batch}
    if call == "serve":
        # requests arrive mixed: a fixed shuffle of the sizes
        members = _members(case)
        order = sorted(range(len(members)), key=lambda i: _spread(i, 0.7548776662466927))
        lists = _member_edges([members[i] for i in order], seed)
        return {"call": call, "requests": [(n, s.cpu().numpy(), d.cpu().numpy()) for n, s, d in lists],
                "server": H.Server(hbm_budget_bytes=64 << 30)}
    n = case["n"]
    src, dst = _graph(case["family"], n, case["k"], seed)
    if call == "partitioned":
        return {"call": call, "n": n, "src": src.cpu().numpy(), "dst": dst.cpu().numpy(),
                "budget": case["budget_mb"] << 20}
    if call == "edges":
        if case["host"]:
            src, dst = src.cpu().numpy(), dst.cpu().numpy()
        return {"call": call, "n": n, "src": src, "dst": dst}
    g = H.harp_build_csr(n, src, dst)
    state = {"call": call, "g": g}
    if call == "literal":
        plan = H.harp_plan()
        plan.version, plan.basis = H.HARP_ABI_VERSION, H.HARP_BASIS_LITERAL
        state["plan"] = plan
    if call == "orbits":
        state["out"] = torch.zeros(n, H.HARP_NORBITS, dtype=torch.int64, device=DEV)
    if call == "edge_orbits":
        # room for every input pair (a fixed shape); rows past the graph's m edges stay zero
        state["out"] = torch.zeros(src.numel(), H.HARP_NEDGE_ORBITS, dtype=torch.int64, device=DEV)
    return state


def run(state):
    call = state["call"]
    if call == "count":
        return H.harp_count4(state["g"]).view(np.int64)
    if call == "edges":
        return H.count4_edges(state["n"], state["src"], state["dst"]).view(np.int64)
    if call == "batch":
        return H.harp_batch_count(state["batch"]).view(np.int64)
    if call == "orbits":
        return H.harp_count4_orbits(state["g"], state["out"])
    if call == "edge_orbits":
        return H.harp_count4_edge_orbits(state["g"], state["out"])
    if call == "literal":
        return H.harp_count4(state["g"], state["plan"]).view(np.int64)
    if call == "serve":
        server = state["server"]
        tickets = [server.submit(n, src, dst) for n, src, dst in state["requests"]]
        return np.stack([server.wait(t, 60_000.0) for t in tickets]).view(np.int64)
    counts, _ = H.harp_count4_partitioned(state["n"], state["src"], state["dst"], state["budget"])
    return counts.view(np.int64)


def work(case):
    """Each input read once (the CSR of a handle: 8 (n + 1) + 8 m bytes; an edge list: 8 m) and each output
    written once.  There are no floating-point operations."""
    call = case["call"]
    if call in ("batch", "serve"):
        members = _members(case)
        n, m = sum(x[1] for x in members), sum(x[1] * x[2] / 2 for x in members)
        return {"bytes": 8 * m + (8 * (n + len(members)) if call == "batch" else 0) + 48 * len(members), "flops": 0}
    n, m = case["n"], case["n"] * case["k"] / 2
    if call in ("edges", "partitioned"):
        return {"bytes": 8 * m + 48, "flops": 0}
    out = {"orbits": 8 * H.HARP_NORBITS * n, "edge_orbits": 8 * H.HARP_NEDGE_ORBITS * m}.get(call, 48)
    return {"bytes": 8 * (n + 1) + 8 * m + out, "flops": 0}


def exact(case, seed):
    """The six counts from the dense adjacency matrix, where that is quick; None elsewhere."""
    if case["call"] not in ("count", "edges", "literal") or case["n"] > 8192:
        return None
    n = case["n"]
    src, dst = _graph(case["family"], n, case["k"], seed)
    A = torch.zeros(n, n, dtype=torch.float64, device=DEV)
    A[src.long(), dst.long()] = 1.0
    A[dst.long(), src.long()] = 1.0
    A.fill_diagonal_(0.0)
    A2 = A @ A                                   # walks of length two: common neighbours off the diagonal
    d = A.sum(1)
    t = A2 * A                                   # t_e at every adjacent pair
    tv = t.sum(1) / 2                            # triangles through each vertex
    T = tv.sum() / 3
    off = A2 - torch.diag(torch.diagonal(A2))
    c4 = (off * (off - 1) / 2).sum() / 4         # each 4-cycle has two opposite pairs, each pair twice
    D = (t * (t - 1) / 2 * A).sum() / 2
    k4 = torch.zeros((), dtype=torch.float64, device=DEV)
    for v in torch.nonzero(tv >= 3).flatten().tolist():
        nb = torch.nonzero(A[v]).flatten()
        nb = nb[nb > v]                          # each 4-clique once, at its lowest vertex
        if nb.numel() >= 3:
            B = A[nb][:, nb]
            k4 += ((B @ B) * B).sum() / 6
    S = (d * (d - 1) * (d - 2) / 6).sum()
    P = (A * torch.outer(d - 1, d - 1)).sum() / 2 - 3 * T
    paw = (tv * (d - 2)).sum()
    diamond = D - 6 * k4
    cycle = c4 - diamond - 3 * k4
    paw = paw - 4 * diamond - 12 * k4
    path = P - 2 * paw - 4 * cycle - 6 * diamond - 12 * k4
    star = S - paw - 2 * diamond - 4 * k4
    return np.array([round(float(v)) for v in (star, path, paw, cycle, diamond, k4)], dtype=np.int64)

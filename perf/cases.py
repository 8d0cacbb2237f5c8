"""What the performance of this library is measured on.

A case is one call a program makes: the coreness of one graph (the convenience
call, synchronised and checked as by default), of a packed batch of graphs, of
a graph just validated, or of a graph kept under batches of edge insertions
and deletions. Graphs are made on the device from the seed alone: R-MAT
(social and web graphs), Chung-Lu with a planted clique (hubs of very high
degree and many levels), Erdos-Renyi (no skew) and 4-neighbour grids (road-like,
one level with very long chains). `relabel` permutes the vertex ids, as files
whose ids say nothing about degree do.
"""
from __future__ import annotations

import math

import torch

import paper_2402_15253_gb300 as pico

RMAT_ABC = (0.57, 0.19, 0.19)
CLIQUE = 3000           # planted clique of the large Chung-Lu graphs
EXACT_MAX_ARCS = 1 << 27


def listed():
    return [
        # an ego network or a small community: latency and launches are all there is
        {"name": "rmat10-peelone", "kind": "single", "family": "rmat", "scale": 10, "ef": 16,
         "off": 32, "algo": "peelone", "relabel": False},
        # a small social graph with the method left to the library
        {"name": "rmat16-auto", "kind": "single", "family": "rmat", "scale": 16, "ef": 16,
         "off": 32, "algo": "auto", "relabel": False},
        # a mid-size graph without skew, odd vertex count, 64-bit offsets
        {"name": "er300k-peelone", "kind": "single", "family": "er", "n": 300007, "deg": 16,
         "off": 64, "algo": "peelone", "relabel": False},
        # a graph from outside, arbitrary ids: checked first, then decomposed
        {"name": "ingest-rmat20", "kind": "ingest", "family": "rmat", "scale": 20, "ef": 16,
         "off": 32, "algo": "auto", "relabel": True},
        # the usual mid-size web graph
        {"name": "rmat22-peelone", "kind": "single", "family": "rmat", "scale": 22, "ef": 16,
         "off": 64, "algo": "peelone", "relabel": False},
        # a crawl with a few enormous hubs and arbitrary ids, by the default method
        {"name": "chunglu22-peelone", "kind": "single", "family": "chunglu", "n": (1 << 22) + 3,
         "ppv": 10, "off": 32, "algo": "peelone", "relabel": True},
        # the same shape at the largest size, method left to the library
        {"name": "chunglu24-auto", "kind": "single", "family": "chunglu", "n": 1 << 24,
         "ppv": 10, "off": 32, "algo": "auto", "relabel": False},
        # a road-like network: hardly any parallelism, thousands of dependent steps
        {"name": "grid4096-peelone", "kind": "single", "family": "grid", "rows": 4096,
         "cols": 4096, "off": 32, "algo": "peelone", "relabel": False},
        # the large social graph, by each method
        {"name": "rmat24-peelone", "kind": "single", "family": "rmat", "scale": 24, "ef": 16,
         "off": 32, "algo": "peelone", "relabel": False},
        {"name": "rmat24-histocore", "kind": "single", "family": "rmat", "scale": 24, "ef": 16,
         "off": 32, "algo": "histocore", "relabel": False},
        # a thousand graphs of 100 to 200,000 vertices solved at once
        {"name": "batch1024", "kind": "batch", "graphs": 1024, "nmin": 100, "nmax": 200000,
         "algo": "peelone"},
        # a graph under a stream of edges: 10,000 arrive, later the same ones leave
        {"name": "maintain-rmat22", "kind": "maintain", "family": "rmat", "scale": 22, "ef": 16,
         "off": 64, "batch": 10000, "relabel": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("single",) * 5 + ("batch", "maintain", "ingest"))
    if kind == "batch":
        nmax = _log_int(rng, 400, 200000)
        graphs = min(_log_int(rng, 16, 8192), int(2.5e7 / nmax * math.log(nmax / 50)) + 16)
        return {"kind": kind, "graphs": graphs, "nmin": rng.randint(20, 100), "nmax": nmax,
                "algo": rng.choice(("peelone", "auto"))}
    family = rng.choice(("rmat", "rmat", "chunglu", "er", "grid") if kind == "single"
                        else ("rmat", "chunglu", "er"))
    case = {"kind": kind, "family": family, "off": rng.choice((32, 64)),
            "relabel": rng.random() < 0.5}
    big = kind == "single"
    if family == "rmat":
        case.update(scale=rng.randint(9, 23 if big else 21), ef=rng.randint(4, 24))
    elif family == "chunglu":
        case.update(n=_log_int(rng, 3000, 6000000 if big else 1000000) | 1, ppv=rng.randint(4, 12))
    elif family == "er":
        n = _log_int(rng, 1000, 8000000 if big else 1000000) | 1
        case.update(n=n, deg=min(rng.randint(3, 40), int(1.2e8 / n)))
    else:
        case.update(rows=_log_int(rng, 20, 4000), cols=_log_int(rng, 20, 4000) | 1)
    if kind == "maintain":
        case["batch"] = _log_int(rng, 50, 5000)
    else:
        # the index method on a grid needs as many rounds as the grid is wide:
        # nobody picks it there
        case["algo"] = rng.choice(("peelone", "auto") if family == "grid"
                                  else ("peelone", "histocore", "auto"))
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _rmat_pairs(scale, count, gen):
    """count endpoint pairs: one quadrant of the 2 x 2 recursive matrix per bit."""
    a, b, c = RMAT_ABC
    src = torch.zeros(count, dtype=torch.int64, device="cuda")
    dst = torch.zeros(count, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        r = torch.rand(count, device="cuda", generator=gen)
        src = (src << 1) | (r >= a + b)
        dst = (dst << 1) | (((r >= a) & (r < a + b)) | (r >= a + b + c))
    return src, dst


def _chunglu_pairs(n, count, gen):
    """count pairs, both ends proportional to (i + 1)^(-1 / 1.1)."""
    # summed on the host, in order: the same thresholds every time
    cdf = torch.cumsum(torch.arange(1, n + 1, dtype=torch.float64) ** (-1 / 1.1), 0)
    cdf = (cdf / cdf[-1].clone()).cuda()
    ends = []
    for _ in range(2):
        r = torch.rand(count, dtype=torch.float64, device="cuda", generator=gen)
        ends.append(torch.searchsorted(cdf, r, right=True).clamp_(max=n - 1))
    return ends


def _er_pairs(n, count, gen):
    return (torch.randint(n, (count,), device="cuda", generator=gen),
            torch.randint(n, (count,), device="cuda", generator=gen))


def _in_chunks(make, total, n):
    """Undirected edge keys lo * n + hi of `total` samples, drawn piece by piece."""
    keys, step = [], 1 << 26
    for first in range(0, total, step):
        s, d = make(min(step, total - first))
        keep = s != d
        keys.append((torch.minimum(s, d) * n + torch.maximum(s, d))[keep])
    return torch.cat(keys)


def _csr(keys, n, off, perm=None):
    """Sorted simple CSR of undirected edge keys, both arc directions stored."""
    if perm is not None:
        a, b = perm[keys // n], perm[keys % n]
        keys = torch.minimum(a, b) * n + torch.maximum(a, b)
        del a, b
    keys = torch.unique(keys)
    lo, hi = keys // n, keys % n
    del keys
    arcs = torch.sort(torch.cat([lo * n + hi, hi * n + lo])).values
    del lo, hi
    rows = torch.arange(n + 1, dtype=torch.int64, device="cuda") * n
    row_ptr = torch.searchsorted(arcs, rows)
    col = (arcs % n).to(torch.int32)
    return row_ptr.to(torch.int64 if off == 64 else torch.int32), col


def _vertices(case):
    if case["family"] == "rmat":
        return 1 << case["scale"]
    if case["family"] == "grid":
        return case["rows"] * case["cols"]
    return case["n"]


def _pairs(case):
    """Undirected edges sampled (a few are dropped as duplicates or loops)."""
    if case["family"] == "rmat":
        return case["ef"] << case["scale"]
    if case["family"] == "chunglu":
        c = _clique(case)
        return case["ppv"] * case["n"] + c * (c - 1) // 2
    if case["family"] == "er":
        return case["n"] * case["deg"] // 2
    return case["rows"] * (case["cols"] - 1) + (case["rows"] - 1) * case["cols"]


def _clique(case):
    return min(CLIQUE, case["n"] // 100)


def _graph(case, gen):
    n = _vertices(case)
    if case["family"] == "grid":
        ids = torch.arange(n, dtype=torch.int64, device="cuda").view(case["rows"], case["cols"])
        keys = torch.cat([(ids[:, :-1] * n + ids[:, 1:]).reshape(-1),
                          (ids[:-1] * n + ids[1:]).reshape(-1)])
        # a map has holes: one crossing in a thousand is missing
        hole = torch.zeros(n, dtype=torch.bool, device="cuda")
        hole[torch.randperm(n, device="cuda", generator=gen)[:max(3, n // 1000)]] = True
        keys = keys[~(hole[keys // n] | hole[keys % n])]
    elif case["family"] == "rmat":
        keys = _in_chunks(lambda c: _rmat_pairs(case["scale"], c, gen), _pairs(case), n)
    elif case["family"] == "er":
        keys = _in_chunks(lambda c: _er_pairs(n, c, gen), _pairs(case), n)
    else:
        keys = _in_chunks(lambda c: _chunglu_pairs(n, c, gen), case["ppv"] * n, n)
        members = torch.randperm(n, device="cuda", generator=gen)[:_clique(case)].sort().values
        i, j = torch.triu_indices(members.numel(), members.numel(), 1, device="cuda")
        keys = torch.cat([keys, members[i] * n + members[j]])
    perm = torch.randperm(n, device="cuda", generator=gen) if case["relabel"] else None
    return _csr(keys, n, case["off"], perm)


def _batch(case, gen):
    """A packed batch: sizes spread log-uniformly (the same for every seed), even
    graphs Erdos-Renyi of mean degree 4 to 64, odd ones R-MAT of edge factor 8
    to 32 cut at their vertex count."""
    G = case["graphs"]
    u = torch.rand(2, G, dtype=torch.float64, generator=torch.Generator().manual_seed(
        int(torch.randint(1 << 31, (1,), device="cuda", generator=gen))))
    at = torch.rand(G, dtype=torch.float64, generator=torch.Generator().manual_seed(G))
    n = torch.exp(math.log(case["nmin"]) + at * math.log(case["nmax"] / case["nmin"]))
    n = n.round().to(torch.int64)
    er = torch.arange(G) % 2 == 0
    count = torch.where(er, n.double() * (4 + 60 * u[0]) / 2,
                        n.double() * torch.floor(8 + 25 * u[1])).to(torch.int64)
    voff = torch.zeros(G + 1, dtype=torch.int64)
    voff[1:] = torch.cumsum(n, 0)
    total = int(voff[-1])
    owner = torch.repeat_interleave(torch.arange(G), count).cuda()
    nd, vd = n.cuda(), voff.cuda()
    nn = nd[owner]
    s = (torch.rand(owner.numel(), dtype=torch.float64, device="cuda", generator=gen) * nn).long()
    d = (torch.rand(owner.numel(), dtype=torch.float64, device="cuda", generator=gen) * nn).long()
    for bits in range(1, int(n.max() - 1).bit_length() + 1):   # the R-MAT graphs, by scale
        sel = (~er) & (n > 1 << (bits - 1)) & (n <= 1 << bits)
        at = torch.nonzero(sel.cuda()[owner]).view(-1)
        if at.numel():
            s[at], d[at] = _rmat_pairs(bits, at.numel(), gen)
    keep = (s < nn) & (d < nn) & (s != d)
    base = vd[owner]
    del owner, nn
    lo, hi = torch.minimum(s, d)[keep], torch.maximum(s, d)[keep]
    base = base[keep]
    rp, col = _csr((lo + base) * total + hi + base, total, 64)
    del lo, hi, s, d, base, keep
    aoff = rp[vd]                                   # first arc of each graph
    arc_owner = torch.repeat_interleave(torch.arange(G, device="cuda"), aoff[1:] - aoff[:-1])
    col -= vd[arc_owner].to(torch.int32)            # graph-local ids
    del arc_owner
    vtx_owner = torch.repeat_interleave(torch.arange(G, device="cuda"), nd)
    local = torch.empty(total + G, dtype=torch.int32, device="cuda")
    local[torch.arange(total, device="cuda") + vtx_owner] = (rp[:-1] - aoff[vtx_owner]).to(torch.int32)
    local[vd[1:] + torch.arange(G, device="cuda")] = (aoff[1:] - aoff[:-1]).to(torch.int32)
    return vd, aoff, local, col


def _new_edges(rp, ci, n, count, gen):
    """count distinct undirected edges that the graph does not have."""
    rp = rp.to(torch.int64)
    s, d = _er_pairs(n, 2 * count + 64, gen)
    lo, hi = torch.minimum(s, d), torch.maximum(s, d)
    first, last = rp[lo], rp[lo + 1]
    for _ in range(32):                             # binary search of hi in lo's sorted row
        mid = (first + last) // 2
        go = (first < last) & (ci[mid.clamp(max=ci.numel() - 1)] < hi)
        first, last = torch.where(go, mid + 1, first), torch.where(go | (first >= last), last, mid)
    found = (first < rp[lo + 1]) & (ci[first.clamp(max=ci.numel() - 1)] == hi)
    keys = torch.unique((lo * n + hi)[(lo != hi) & ~found])
    keys = keys[torch.randperm(keys.numel(), device="cuda", generator=gen)[:count]]
    return torch.stack([keys // n, keys % n], 1).to(torch.int32)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if case["kind"] == "batch":
        vo, ao, rp, ci = _batch(case, gen)
        return {"case": case, "vo": vo, "ao": ao, "rp": rp, "ci": ci, "tv": int(vo[-1]),
                "ta": int(ao[-1])}
    rp, ci = _graph(case, gen)
    state = {"case": case, "rp": rp, "ci": ci}
    if case["kind"] == "maintain":
        state["edges"] = _new_edges(rp, ci, rp.numel() - 1, case["batch"], gen)
        state["graph"] = pico.DynamicGraph(rp, ci, capacity_arcs=ci.numel() + 4 * case["batch"])
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        return pico.coreness_batched(state["vo"], state["ao"], state["rp"], state["ci"],
                                     case["algo"], total_vertices=state["tv"],
                                     total_arcs=state["ta"])
    rp, ci = state["rp"], state["ci"]
    if case["kind"] == "maintain":
        g = state["graph"]
        g.update(insert=state["edges"])
        arrived = g.coreness()
        g.update(delete=state["edges"])
        return arrived, g.coreness()
    if case["kind"] == "ingest":   # a graph from outside: checked, then decomposed
        check = pico.pico_validate_graph if rp.dtype == torch.int32 else pico.pico_validate_graph_i64
        status, defects = check(rp, ci, rp.numel() - 1, ci.numel())
        return status, defects, pico.coreness(rp, ci, case["algo"])
    return pico.coreness(rp, ci, case["algo"])


def _size(case):
    """(vertices, arcs) of a case, arcs as sampled."""
    if case["kind"] == "batch":
        lo, hi = case["nmin"], case["nmax"]
        n = case["graphs"] * (hi - lo) / max(math.log(hi / lo), 1e-9)
        return n, n * (34 + 40) / 2
    return _vertices(case), 2 * _pairs(case)


def work(case):
    """Row offsets and columns read once, coreness written once; an update
    reads the graph's rows once and its batch, and writes the new rows."""
    n, m = _size(case)
    w = 4 if case.get("off", 32) == 32 else 8
    if case["kind"] == "maintain":
        return {"bytes": 2 * (2 * (8 * n + 4 * m) + 4 * n + 8 * case["batch"]), "flops": 0}
    return {"bytes": w * (n + 1) + 4 * m + 4 * n, "flops": 0}


# ---------------------------------------------------------------------------
# the coreness by definition, in plain torch
# ---------------------------------------------------------------------------

def _peel(rp, ci):
    """Removes the vertices of smallest residual degree, level by level."""
    rp = rp.to(torch.int64)
    deg = rp[1:] - rp[:-1]
    core = torch.zeros_like(deg)
    left = torch.nonzero(deg > 0).view(-1)
    k = 0
    deg = deg.clone()
    while left.numel():
        k = max(k, int(deg[left].min()))
        gone = deg[left] <= k
        front, left = left[gone], left[~gone]
        core[front] = k
        deg[front] = -1 << 40
        cnt = rp[front + 1] - rp[front]
        first = torch.repeat_interleave(rp[front] - torch.cumsum(cnt, 0) + cnt, cnt)
        nbr = ci[first + torch.arange(first.numel(), device=first.device)].long()
        deg.index_add_(0, nbr, torch.full_like(nbr, -1))
    return core


def exact(case, seed):
    n, m = _size(case)
    if m > EXACT_MAX_ARCS or (case["kind"] != "batch" and case["family"] == "grid" and n > 1 << 20):
        return None
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if case["kind"] == "batch":
        vo, ao, rp, ci = _batch(case, gen)
        G = vo.numel() - 1
        owner = torch.repeat_interleave(torch.arange(G, device="cuda"), vo[1:] - vo[:-1])
        whole = torch.empty(int(vo[-1]) + 1, dtype=torch.int64, device="cuda")
        whole[:-1] = rp[torch.arange(owner.numel(), device="cuda") + owner] + ao[owner]
        whole[-1] = ao[-1]
        col = ci + torch.repeat_interleave(vo[:-1], ao[1:] - ao[:-1])
        return _peel(whole, col)
    rp, ci = _graph(case, gen)
    if case["kind"] == "maintain":
        nv = rp.numel() - 1
        e = _new_edges(rp, ci, nv, case["batch"], gen).long()
        row = torch.repeat_interleave(torch.arange(nv, device="cuda"), (rp[1:] - rp[:-1]).long())
        keys = torch.cat([(row * nv + ci)[row < ci], e[:, 0] * nv + e[:, 1]])
        return _peel(*_csr(keys, nv, 64)), _peel(rp, ci)
    if case["kind"] == "ingest":
        return 0, 0, _peel(rp, ci)
    return _peel(rp, ci)

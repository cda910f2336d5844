"""What users of the framework have it do, as cases that can be timed and compared.

Every case builds a seeded synthetic graph (R-MAT with the quadrant weights
0.57 / 0.19 / 0.19, or the community graph: blocks of 1024 vertices, Zipf(2)
out-degrees, 90 % of the edges inside the block), as a symmetric CSR with
strictly increasing rows, and makes one call of the public API on it.

  pagerank   lg_pagerank on an encoded graph
  bfs        lg_bfs from `sources` sources on an encoded graph
  sssp       lg_sssp from one source on an encoded weighted graph
  neighbors  lg_neighbors: `k` random vertices looked up
  encode     lg_encode of a CSR that is in device memory
  decode     lg_decode of the whole graph
  batch      lg_batch_run: encode + BFS + PageRank of many small graphs
  serve      lg_server_replay of a burst of mixed requests (host data in, host data out)

The shape of a case's graph (its edges up to the vertex labels) belongs to the
case; the seed gives the labels, the weights, the sources and the requests'
vertices.  So every seed has other arrays of the same sizes.
"""
import math

import numpy as np
import torch

import paper_2010_15879_gb300 as lg

IDS = {"global": lg.LG_ID_GLOBAL, "local": lg.LG_ID_LOCAL, "gap": lg.LG_ID_LOCAL_GAP, "csr32": lg.LG_ID_CSR32}
OFFS = {"packed": lg.LG_OFF_PACKED, "ef": lg.LG_OFF_EF}
RELABEL = {"none": lg.LG_RELABEL_NONE, "dm": lg.LG_RELABEL_DM}
DAMPING = 0.85
BLOCK = 1024          # vertices of a community block
ZIPF_MAX = 1 << 14
ROWS_AT_ONCE = 1 << 28  # arcs sorted at a time


# --- graphs -----------------------------------------------------------------

def _rng(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + stream)
    return g


def _labels(n, seed):
    """The seed's labels of the vertices 0 .. n - 1 of a shape."""
    return torch.randperm(n, generator=_rng(seed + 1, 1), device="cuda", dtype=torch.int32)


def _rmat_edges(n, ef, seed):
    """Endpoints of ef * 2^ceil(log2 n) R-MAT edges; those with an endpoint not
    below n are for the caller to drop."""
    scale = max(1, (n - 1).bit_length())
    m, rng = ef << scale, _rng(0, 1)
    perm = torch.randperm(1 << scale, generator=rng, device="cuda", dtype=torch.int32)
    inside = perm < n
    perm[inside] = _labels(n, seed)[perm[inside]]
    u = torch.empty(m, dtype=torch.int32, device="cuda")
    v = torch.empty(m, dtype=torch.int32, device="cuda")
    step = 1 << 27
    for a in range(0, m, step):
        b = min(m, a + step)
        x = torch.zeros(b - a, dtype=torch.int32, device="cuda")
        y = torch.zeros(b - a, dtype=torch.int32, device="cuda")
        for _ in range(scale):
            r = torch.rand(b - a, generator=rng, device="cuda")
            x.mul_(2).add_(r >= 0.76)
            y.mul_(2).add_((r >= 0.95) | ((r >= 0.57) & (r < 0.76)))
        u[a:b] = perm[x]
        v[a:b] = perm[y]
    return u, v


def _community_edges(n, seed):
    """Endpoints of the community graph's edges (mean out-degree 16)."""
    rng = _rng(0, 2)
    p = torch.arange(1, ZIPF_MAX + 1, dtype=torch.float64, device="cuda").pow(-2.0)
    mean = float((p * torch.arange(1, ZIPF_MAX + 1, dtype=torch.float64, device="cuda")).sum() / p.sum())
    cdf = torch.cumsum(p / p.sum(), 0)
    z = torch.searchsorted(cdf, torch.rand(n, generator=rng, device="cuda", dtype=torch.float64)) + 1
    deg = (z.clamp(max=ZIPF_MAX).double() * (16.0 / mean)).round().clamp(min=1).long()
    u = torch.repeat_interleave(torch.arange(n, dtype=torch.int32, device="cuda"), deg)
    m = u.numel()
    base = (u // BLOCK) * BLOCK
    size = (n - base).clamp(max=BLOCK)
    step = (torch.rand(m, generator=rng, device="cuda", dtype=torch.float64) * (size - 1)).int() + 1
    inside = base + (u - base + step) % size
    anywhere = (torch.rand(m, generator=rng, device="cuda", dtype=torch.float64) * n).int()
    v = torch.where(torch.rand(m, generator=rng, device="cuda") < 0.9, inside, anywhere)
    perm = _labels(n, seed)
    return perm[u], perm[v]


def _csr(n, u, v):
    """Symmetric CSR without self loops or repeated arcs: row_ptr int64, col int32."""
    parts = max(1, math.ceil(2 * u.numel() / ROWS_AT_ONCE))
    cols, ptrs, at = [], [], 0
    for k in range(parts):
        lo, hi = n * k // parts, n * (k + 1) // parts
        keys = []
        for a, b in ((u, v), (v, u)):
            keep = (a >= lo) & (a < hi) & (b < n) & (a != b)
            keys.append((a[keep].long() << 32) | b[keep].long())
        keys = torch.unique(torch.cat(keys))
        ptrs.append(torch.searchsorted(keys, torch.arange(lo, hi, device="cuda") << 32) + at)
        at += keys.numel()
        cols.append((keys & 0xFFFFFFFF).int())
        del keys
    ptrs.append(torch.tensor([at], device="cuda"))
    return torch.cat(ptrs), torch.cat(cols)


def _weights(n, rp, col, seed):
    """Uniform integer weights in [1, 255], the same for an arc and its reverse."""
    out = torch.empty_like(col)
    parts = max(1, math.ceil(col.numel() / ROWS_AT_ONCE))
    for k in range(parts):
        lo, hi = n * k // parts, n * (k + 1) // parts
        a, b = int(rp[lo]), int(rp[hi])
        row = torch.repeat_interleave(torch.arange(lo, hi, device="cuda"), rp[lo + 1:hi + 1] - rp[lo:hi])
        other = col[a:b].long()
        h = torch.minimum(row, other) * 0x9E3779B1 + torch.maximum(row, other) * 0x85EBCA77 + (int(seed) + 1) * 0xC2B2AE3D
        h = (h ^ (h >> 29)) * 0x27D4EB2F
        out[a:b] = (((h ^ (h >> 31)) & 0x7FFFFFFF) % 255 + 1).int()
    return out


def _graph(case, seed):
    u, v = _rmat_edges(case["n"], case["ef"], seed) if case["graph"] == "rmat" else _community_edges(case["n"], seed)
    rp, col = _csr(case["n"], u, v)
    del u, v
    w = _weights(case["n"], rp, col, seed) if case.get("weighted") else None
    if col.numel() > ROWS_AT_ONCE:
        torch.cuda.empty_cache()  # the library's own pool shares the card
    return rp, col, w


def _options(case):
    return {"id_mode": IDS[case["ids"]], "off_mode": OFFS[case["off"]], "relabel": RELABEL[case["relabel"]],
            "weight_bits": 8 if case.get("weighted") else 0}


def _sources(rp, k, seed):
    """k random vertices of nonzero degree."""
    nz = torch.nonzero(rp[1:] > rp[:-1]).flatten()
    return nz[torch.randint(nz.numel(), (k,), generator=_rng(seed, 3), device="cuda")].int()


def _batch_input(case, seed):
    """graph_vptr, row_ptr, col of `graphs` R-MAT graphs: scales log-uniform in
    [8, 16], edge factors in [4, 32]; col holds IDs local to the graph."""
    host = np.random.default_rng(case["graphs"])
    scale = torch.from_numpy(np.floor(host.uniform(8, 17, case["graphs"])).astype(np.int64)).cuda()
    ef = torch.from_numpy(host.integers(4, 33, case["graphs"])).cuda()
    vptr = torch.zeros(case["graphs"] + 1, dtype=torch.int64, device="cuda")
    vptr[1:] = torch.cumsum(1 << scale, 0)
    g = torch.repeat_interleave(torch.arange(case["graphs"], dtype=torch.int32, device="cuda"), ef << scale)
    s, rng = scale.int()[g], _rng(0, 4)
    x, y = torch.zeros_like(s), torch.zeros_like(s)
    for level in range(16):
        r = torch.rand(s.numel(), generator=rng, device="cuda")
        on = s > level
        x = torch.where(on, 2 * x + (r >= 0.76).int(), x)
        y = torch.where(on, 2 * y + ((r >= 0.95) | ((r >= 0.57) & (r < 0.76))).int(), y)
    label = torch.randint(1 << 14, (2, case["graphs"]), generator=_rng(seed, 4), device="cuda", dtype=torch.int32)
    mask, mul, add = (1 << s) - 1, 2 * label[0][g] + 1, label[1][g]
    x, y = (x * mul + add) & mask, (y * mul + add) & mask  # the seed's labels of each graph
    V, base = int(vptr[-1]), vptr[g.long()]
    rp, col = _csr(V, (base + x).int(), (base + y).int())
    owner = torch.repeat_interleave(torch.arange(case["graphs"], device="cuda"), rp[vptr[1:]] - rp[vptr[:-1]])
    return vptr, rp, (col - vptr[owner]).int()


def _serve_input(case, seed):
    """Three CSRs of n, n/4 and n/16 vertices and a burst of requests: 60 %
    lookups of 1 to 256 vertices, 30 % BFS, 10 % personalized PageRank."""
    csrs = [_graph({"graph": "rmat", "n": case["n"] >> (2 * k), "ef": 16}, seed)[:2] for k in range(3)]
    labels = [_labels(case["n"] >> (2 * k), seed).cpu().numpy() for k in range(3)]
    host, R = np.random.default_rng(case["requests"]), case["requests"]
    kind = np.array([0, 0, 0, 0, 0, 0, 1, 1, 1, 2], dtype=np.uint32)[np.arange(R) % 10]
    kind = host.permutation(kind)
    graph = host.integers(0, 3, R).astype(np.uint32)
    sources = [_sources(rp, R, seed).cpu().numpy() for rp, _ in csrs]
    source = np.array([sources[graph[i]][i] for i in range(R)], dtype=np.uint32)
    count = np.where(kind == 0, host.integers(1, 257, R), 0)
    off = np.concatenate([[0], np.cumsum(count)]).astype(np.uint64)
    ids = np.concatenate([labels[graph[i]][host.integers(0, labels[graph[i]].size, count[i])] for i in range(R)])
    return csrs, kind, graph, source, off, ids.astype(np.uint32)


# --- the cases --------------------------------------------------------------

def listed():
    return [
        # One small graph ranked: launches and the last wave count.
        {"name": "pagerank_rmat16", "kind": "pagerank", "graph": "rmat", "n": 65536, "ef": 16, "ids": "global", "off": "packed", "relabel": "none", "iters": 20},
        # Distances from many sources on a small graph: one latency per level.
        {"name": "bfs_rmat16_64src", "kind": "bfs", "graph": "rmat", "n": 65536, "ef": 16, "ids": "global", "off": "packed", "relabel": "none", "sources": 64},
        # One lookup request of a service on a resident graph.
        {"name": "neighbors_rmat20_200", "kind": "neighbors", "graph": "rmat", "n": 1000003, "ef": 16, "ids": "global", "off": "ef", "relabel": "dm", "k": 200},
        # A community graph of ordinary size put into its smallest form.
        {"name": "encode_community_1p5m", "kind": "encode", "graph": "community", "n": 1500007, "ef": 16, "ids": "gap", "off": "ef", "relabel": "dm"},
        # The same kind of graph read back whole.
        {"name": "decode_community_4m", "kind": "decode", "graph": "community", "n": 4000037, "ef": 16, "ids": "gap", "off": "ef", "relabel": "dm"},
        # A social network's communities ranked in compressed form.
        {"name": "pagerank_community_2p24", "kind": "pagerank", "graph": "community", "n": 1 << 24, "ef": 16, "ids": "gap", "off": "ef", "relabel": "dm", "iters": 10},
        # A web-scale graph ranked, weights stored beside the IDs.
        {"name": "pagerank_rmat26", "kind": "pagerank", "graph": "rmat", "n": 1 << 26, "ef": 16, "ids": "global", "off": "ef", "relabel": "dm", "weighted": True, "iters": 10},
        # Distances on a large graph from a handful of sources at once.
        {"name": "bfs_rmat25_16src", "kind": "bfs", "graph": "rmat", "n": 30000001, "ef": 16, "ids": "global", "off": "ef", "relabel": "dm", "weighted": True, "sources": 16},
        # The largest construction: relabel, sort and pack two billion weighted arcs.
        {"name": "encode_rmat26", "kind": "encode", "graph": "rmat", "n": 1 << 26, "ef": 16, "ids": "global", "off": "ef", "relabel": "dm", "weighted": True},
        # Weighted shortest paths on a graph of ordinary size.
        {"name": "sssp_rmat22", "kind": "sssp", "graph": "rmat", "n": 1 << 22, "ef": 16, "ids": "global", "off": "ef", "relabel": "dm", "weighted": True},
        # A thousand small graphs through encode, BFS and PageRank in one launch.
        {"name": "batch_1000", "kind": "batch", "graphs": 1000, "iters": 10},
        # A burst of mixed requests to a server of three resident graphs.
        {"name": "serve_rmat20_120", "kind": "serve", "n": 1000000, "requests": 120},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pagerank", "pagerank", "bfs", "bfs", "encode", "encode", "decode", "neighbors", "sssp", "batch", "serve"])
    if kind == "batch":
        return {"kind": kind, "graphs": _log(rng, 8, 1000), "iters": rng.randint(2, 10)}
    if kind == "serve":
        return {"kind": kind, "n": _log(rng, 20000, 1000000), "requests": rng.randint(20, 120)}
    top = {"pagerank": 25, "bfs": 25, "encode": 25, "decode": 23, "neighbors": 22, "sssp": 22}[kind]
    c = {"kind": kind, "graph": rng.choice(["rmat", "rmat", "community"]) if kind != "sssp" else "rmat", "ef": 16}
    if c["graph"] == "community":
        top = min(top, 24)
    else:
        c["ef"] = rng.randint(8, 24)
    c["n"] = _log(rng, 1 << 12, (1 << top) * 16 // max(16, c["ef"]))
    c["ids"] = "global" if kind == "sssp" else rng.choice(["global", "global", "gap", "local"])
    c["off"] = rng.choice(["ef", "packed"])
    c["relabel"] = rng.choice(["dm", "dm", "none"])
    c["weighted"] = c["ids"] == "global" and (kind == "sssp" or rng.random() < 0.4)
    if kind == "pagerank":
        c["iters"] = rng.randint(1, 20) if c["n"] < 1 << 23 else rng.randint(1, 8)
    if kind == "bfs":
        c["sources"] = _log(rng, 1, 64)
    if kind == "neighbors":
        c["k"] = _log(rng, 1, 4096)
    return c


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        vptr, rp, col = _batch_input(case, seed)
        return {"case": case, "batch": lg.lg_batch_create(vptr, rp, col)}
    if kind == "serve":
        csrs, *trace = _serve_input(case, seed)
        graphs = [lg.lg_encode(rp, col, id_mode=lg.LG_ID_GLOBAL, off_mode=lg.LG_OFF_EF, relabel=lg.LG_RELABEL_DM)
                  for rp, col in csrs]
        rows = [rp.cpu().numpy() for rp, _ in csrs]
        kinds, graph, _, off, ids = trace
        sizes = []
        for i in range(case["requests"]):
            if kinds[i] == lg.LG_REQ_NEIGHBORS:
                vs = ids[int(off[i]):int(off[i + 1])].astype(np.int64)
                r = rows[graph[i]]
                sizes.append(8 * (vs.size + 1) + 4 * int((r[vs + 1] - r[vs]).sum()))
            else:
                sizes.append(4 * (rows[graph[i]].size - 1))
        out = [np.zeros(sum((z + 7) // 8 * 8 for z, k in zip(sizes, kinds) if k == q), dtype=np.uint8) for q in range(3)]
        keep, at = [], [0, 0, 0]
        for z, k in zip(sizes, kinds):
            keep.append(out[k][at[k]:at[k] + z])
            at[k] += (z + 7) // 8 * 8
        server = lg.lg_server_create(graphs, device_bytes=1 << 30, host_bytes=1 << 28)
        return {"case": case, "server": server, "trace": trace, "keep": keep, "out": out,
                "arrival": np.zeros(case["requests"], dtype=np.uint64)}
    rp, col, w = _graph(case, seed)
    if kind == "encode":
        state = {"case": case, "csr": (rp, col, w), "options": _options(case), "graph": None}
        if case["ids"] in ("local", "gap"):  # the lengths of these streams depend on the labels
            n, arcs, s = case["n"], col.numel(), max(1, (case["n"] - 1).bit_length())
            words = {"A": arcs * s + n * (s + 6), "O": 64 * (n + 1) if case["off"] == "packed" else 0}
            words |= {"ef_low": 40 * (n + 1), "ef_high": 3 * (n + 1)} if case["off"] == "ef" else {}
            state["buffers"] = {k: torch.zeros(b // 64 + 8, dtype=torch.int64, device="cuda") for k, b in words.items()}
        return state
    state = {"case": case, "graph": lg.lg_encode(rp, col, w, **_options(case))}
    if kind == "bfs":
        state["sources"] = _sources(rp, case["sources"], seed)
    elif kind == "sssp":
        state["source"] = int(_sources(rp, 1, seed)[0])
    elif kind == "neighbors":
        at = torch.randint(case["n"], (case["k"],), generator=_rng(0, 5), device="cuda")
        state["vertices"] = _labels(case["n"], seed)[at]
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "pagerank":
        return lg.lg_pagerank(state["graph"], DAMPING, case["iters"])
    if kind == "bfs":
        return lg.lg_bfs(state["graph"], state["sources"])
    if kind == "sssp":
        return lg.lg_sssp(state["graph"], state["source"])
    if kind == "neighbors":
        return lg.lg_neighbors(state["graph"], state["vertices"], with_weights=bool(case.get("weighted")))
    if kind == "decode":
        return lg.lg_decode(state["graph"], with_weights=bool(case.get("weighted")))
    if kind == "encode":
        if state["graph"] is not None:
            lg.lg_free_async(state["graph"])
        state["graph"] = lg.lg_encode(*state["csr"], **state["options"])
        out = lg.lg_arrays_device(state["graph"])
        for name, view in out.items():
            view.owner = state["graph"]  # the arrays live as long as the graph
            if name in state.get("buffers", {}):  # kept by the caller, zero behind the stream's end
                state["buffers"][name][:view.numel()].copy_(view)
                out[name] = state["buffers"][name]
        return out
    if kind == "batch":
        return lg.lg_batch_run(state["batch"], DAMPING, case["iters"])
    lg.lg_server_replay(state["server"], *state["trace"], state["arrival"], keep=state["keep"])
    lookups, depths, ranks = state["out"]
    return {"lookups": lookups, "depths": depths.view(np.int32), "ranks": ranks.view(np.float32)}


# --- what a pass cannot do without -------------------------------------------

def _arcs(case):
    """Stored arcs: repeated edges thin an R-MAT graph by 13 % at scale 16 and
    by 1.7 % at scale 27 (edge factor 16)."""
    n = case["n"]
    if case.get("graph", "rmat") == "community":
        return 23.4 * n
    scale, ef = max(1, (n - 1).bit_length()), case.get("ef", 16)
    lost = min(0.5, 0.133 * 0.828 ** (scale - 16) * ef / 16)
    return 2.0 * ef * (1 << scale) * (n / (1 << scale)) ** 2 * (1 - lost)


def _bytes_of(case):
    """Bytes of the encoded graph."""
    n, arcs = case["n"], _arcs(case)
    width = max(1, (n - 1).bit_length())
    if case.get("ids") in ("gap", "local") and case.get("graph") == "community":
        width *= 0.85
    return arcs * (width + (8 if case.get("weighted") else 0)) / 8 + n


def work(case):
    kind = case["kind"]
    if kind == "batch":
        arcs, V = 4.4e5 * case["graphs"], 1.46e4 * case["graphs"]
        sweep = arcs * 14 / 8 + V * 2.5
        return {"bytes": 8 * V + 4 * arcs + sweep * (2 + case["iters"]) + 8 * V * (case["iters"] + 1), "flops": 2.0 * arcs * case["iters"]}
    if kind == "serve":
        n, R = case["n"] * 0.44, case["requests"]  # the mean of the three graphs
        one = {"n": int(n), "ef": 16}
        rows = R * 0.6 * 128 * (8 + 4 * 31)
        return {"bytes": rows + R * 0.4 * 4 * n + R * 0.1 / 8 * 10 * (_bytes_of(one) + 64 * n) + R * 0.3 / 64 * _bytes_of(one),
                "flops": 2.0 * R * 0.1 * 10 * _arcs(one)}
    n, arcs, stream = case["n"], _arcs(case), _bytes_of(case)
    csr = 8 * n + arcs * (8 if case.get("weighted") else 4)
    if kind == "pagerank":
        return {"bytes": case["iters"] * (stream + 8 * n), "flops": 2.0 * arcs * case["iters"]}
    if kind == "bfs":
        return {"bytes": stream + 4.0 * n * case["sources"], "flops": 0}
    if kind == "sssp":
        return {"bytes": stream + 8.0 * n, "flops": 0}
    if kind == "neighbors":
        return {"bytes": case["k"] * (12 + 2 * 4 * arcs / n), "flops": 0}
    return {"bytes": csr + stream, "flops": 0}  # encode, decode: one form in, the other out


# --- the same results in 64 bits ----------------------------------------------

def _ranks64(rp, col, iters, r0, teleport):
    """r_t = teleport + d * sum over neighbors of r_{t-1} / degree."""
    deg = (rp[1:] - rp[:-1]).double()
    inv = torch.where(deg > 0, 1.0 / deg.clamp(min=1), torch.zeros_like(deg))
    r, n, parts = r0, deg.numel(), max(1, math.ceil(col.numel() / ROWS_AT_ONCE))
    cuts = [n * k // parts for k in range(parts + 1)]
    ends = rp[torch.tensor(cuts, device="cuda")].tolist()
    for _ in range(iters):
        c, out = r * inv, torch.empty_like(r)
        for k in range(parts):
            lo, hi, a, b = cuts[k], cuts[k + 1], ends[k], ends[k + 1]
            s = torch.zeros(b - a + 1, dtype=torch.float64, device="cuda")
            torch.cumsum(c[col[a:b]], 0, out=s[1:])
            p = rp[lo:hi + 1] - a
            out[lo:hi] = s[p[1:]] - s[p[:-1]]
        r = teleport + DAMPING * out
    return r


def exact(case, seed):
    kind = case["kind"]
    if kind == "pagerank":
        rp, col, _ = _graph({**case, "weighted": False}, seed)
        n = case["n"]
        one = torch.ones(n, dtype=torch.float64, device="cuda")
        return _ranks64(rp, col, case["iters"], one / n, one * ((1 - DAMPING) / n))
    if kind == "batch":
        vptr, rp, col = _batch_input(case, seed)
        size = vptr[1:] - vptr[:-1]
        own = torch.repeat_interleave(torch.arange(case["graphs"], device="cuda"), size)
        row = torch.repeat_interleave(torch.arange(own.numel(), device="cuda"), rp[1:] - rp[:-1])
        one = 1.0 / size.double()[own]
        return [None, _ranks64(rp, col.long() + vptr[own[row]], case["iters"], one, (1 - DAMPING) * one)]
    if kind == "serve":
        csrs, kinds, graph, source, _, _ = _serve_input(case, seed)
        out = []
        for i in np.nonzero(kinds == lg.LG_REQ_PPR)[0]:
            rp, col = csrs[graph[i]]
            e = torch.zeros(rp.numel() - 1, dtype=torch.float64, device="cuda")
            e[int(source[i])] = 1.0
            r = _ranks64(rp, col, 10, e, (1 - DAMPING) * e)
            out.append(torch.cat([r, torch.zeros(r.numel() % 2, dtype=torch.float64, device="cuda")]))
        return {"lookups": None, "depths": None, "ranks": torch.cat(out) if out else None}
    return None

"""The work that users of the BigGraphVis library have it do, as measured cases.

A case is a dict of plain values.  ``kind`` says which public entry points of
``paper_2108_00529_gb300.bgv`` it goes through:

* ``layout``       the whole pipeline on a device-resident edge list (bgv_layout),
                   or from pinned host buffers (``host``: bgv_layout_host)
* ``batch``        many graphs of uneven size in one call (bgv_layout_batched)
* ``sketch``       the degree count-min sketch of an edge stream
* ``communities``  the streaming community rounds on sketched degrees
* ``supergraph``   relabelling, superedges, masses and CSR from labels
* ``csr``          the whole graph's CSR, for a layout of the graph itself
* ``run``          initial positions and a ForceAtlas2 run on a whole graph
* ``step``         one ForceAtlas2 step of a caller's own loop (an interactive view)
* ``picture``      colour groups, node colours and the drawn image of a layout

Graphs are made on the GPU from the seed alone: R-MAT (skewed degrees, ids not
permuted) or planted partitions (communities of lognormal size, ids permuted).
Sizes follow the repository's workloads: sbm16, rmat20, rmat22x, lnpp1m and
batch512 (graphgen, bench.py).  Output buffers are sized by their upper bounds,
as the library asks, and start as zeros: rows past the supernodes and superedges
found stay zero.
"""
import math

import numpy as np
import torch

from paper_2108_00529_gb300 import bgv as B

RMAT20 = {"graph": "rmat", "scale": 20, "a": 0.57, "b": 0.19}
RMAT22 = {"graph": "rmat", "scale": 22, "a": 0.45, "b": 0.22}


def listed():
    return [
        # a small collaboration graph laid out on request: latency and launches
        {"name": "layout_1k", "kind": "layout", "graph": "planted", "n": 1000, "m": 5000, "k": 8, "intra": 0.8,
         "width": 4096, "threshold": 0, "iterations": 200, "host": False},
        # the small planted-partition workload (sbm16: 16 communities, 200 iterations, threshold 64)
        {"name": "layout_sbm16", "kind": "layout", "graph": "planted", "n": 10_000, "m": 40_283, "k": 16,
         "intra": 0.775, "width": 4096, "threshold": 64, "iterations": 200, "host": False},
        # a social graph of a million ids, device to device (rmat20)
        {"name": "layout_rmat20", "kind": "layout", **RMAT20, "n": 1 << 20, "m": 10_000_000, "width": 65536,
         "threshold": 0, "iterations": 500, "host": False},
        # the paper's largest graph's size, end to end from host buffers (rmat22x, the benchmark workload)
        {"name": "layout_rmat22x_host", "kind": "layout", **RMAT22, "n": 3_200_000, "m": 34_000_000, "width": 65536,
         "threshold": 0, "iterations": 500, "host": True},
        # a collection of graphs laid out together (batch512's size distribution, 160 graphs)
        {"name": "batch_160", "kind": "batch", "graphs": 160, "n_lo": 1000, "n_hi": 200_000, "degree": 10.0,
         "sizes": 1, "width": 4096, "iterations": 300},
        # streaming degree sketch of the largest edge list
        {"name": "sketch_34m", "kind": "sketch", **RMAT22, "n": 3_200_000, "m": 34_000_000, "rows": 4, "width": 65536},
        # community rounds of a skewed graph on its sketched degrees
        {"name": "communities_10m", "kind": "communities", **RMAT20, "n": 1 << 20, "m": 10_000_000, "rows": 4,
         "width": 65536, "passes": 3, "threshold": 0, "tie_mode": 0, "jumps": 0, "mode": 0},
        # supergraph of the largest edge list from its community labels
        {"name": "supergraph_34m", "kind": "supergraph", **RMAT22, "n": 3_200_000, "m": 34_000_000, "rows": 4,
         "width": 65536, "optional": False},
        # whole-graph drawing (the precision form, lnpp1m): CSR, then the 500 iterations
        {"name": "csr_8m", "kind": "csr", "graph": "planted", "n": 1_000_000, "m": 8_000_000, "k": 256, "intra": 0.8},
        {"name": "run_lnpp1m", "kind": "run", "graph": "planted", "n": 1_000_000, "m": 8_000_000, "k": 256,
         "intra": 0.8, "iterations": 500, "theta": 1.2, "strong": 0},
        # one frame of a caller's own loop, odd size
        {"name": "step_60k", "kind": "step", "graph": "planted", "n": 60_013, "m": 300_077, "k": 48, "intra": 0.8,
         "theta": 1.2, "leaf_cap": 1, "strong": 0},
        # the picture: the paper's largest supergraph (248,188 communities), 3.2 M nodes coloured, 2048 x 2048 pixels
        {"name": "picture_248k", "kind": "picture", "K": 248_188, "n": 3_200_000, "W": 2048, "H": 2048},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, n_lo, n_hi):
    """A graph of log-uniform size; odd sizes among them."""
    if rng.random() < 0.4:
        scale = rng.randint(12, 22)
        n = min(n_hi, max(n_lo, int((1 << scale) * rng.uniform(0.55, 1.0)) | 1))
        scale = (n - 1).bit_length()
        deg = rng.uniform(2.0, 10.0)
        a = rng.uniform(0.45, 0.57)
        return {"graph": "rmat", "scale": scale, "a": round(a, 3), "b": round((0.95 - a) / 2, 3), "n": n,
                "m": int(n * deg) | 1}
    n = _log(rng, n_lo, n_hi) | 1
    return {"graph": "planted", "n": n, "m": int(n * rng.uniform(2.0, 10.0)) | 1, "k": _log(rng, 4, max(5, n // 200)),
            "intra": round(rng.uniform(0.6, 0.9), 3)}


def draw(rng):
    kind = rng.choice(["layout", "layout", "batch", "sketch", "communities", "supergraph", "csr", "run", "step",
                       "picture"])
    if kind == "picture":
        return {"kind": kind, "K": _log(rng, 500, 500_000) | 1, "n": _log(rng, 10_000, 3_200_000) | 1,
                "W": rng.randint(400, 3000), "H": rng.randint(400, 3000)}
    if kind == "batch":
        return {"kind": kind, "graphs": _log(rng, 4, 160), "n_lo": 1000, "n_hi": _log(rng, 4000, 200_000),
                "degree": round(rng.uniform(4.0, 10.0), 2), "sizes": rng.randint(2, 1 << 20), "width": 4096,
                "iterations": rng.choice([50, 100, 200, 300])}
    if kind == "step":
        g = _draw_graph(rng, 300, 1_000_000)
        return {"kind": kind, **g, "theta": rng.choice([0.8, 1.0, 1.2]), "leaf_cap": rng.choice([1, 1, 4]),
                "strong": rng.randint(0, 1)}
    g = _draw_graph(rng, 1000, 1_000_000 if kind == "run" else 3_200_000)
    if kind == "layout":
        its = rng.choice([100, 200, 300, 500])
        return {"kind": kind, **g, "width": 65536 if g["m"] > 2_000_000 else 4096,
                "threshold": rng.choice([0, 0, 16, 64]), "iterations": its, "host": rng.random() < 0.5}
    if kind == "run":
        return {"kind": kind, **g, "iterations": rng.choice([50, 100, 200]), "theta": rng.choice([1.0, 1.2]),
                "strong": rng.randint(0, 1)}
    if kind == "csr":
        return {"kind": kind, **g}
    shape = {"rows": rng.randint(2, 6), "width": rng.choice([4096, 5000, 34_500, 65536])}
    if kind == "supergraph":
        return {"kind": kind, **g, **shape, "optional": rng.random() < 0.5}
    if kind == "communities":
        return {"kind": kind, **g, **shape, "passes": rng.randint(1, 10), "threshold": rng.choice([0, 0, 16, 64]),
                "tie_mode": rng.randint(0, 1), "jumps": rng.choice([0, 0, 1]), "mode": rng.choice([0, 0, 1])}
    return {"kind": "sketch", **g, **shape}


# ------------------------------------------------------------------ inputs
def _gen(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(int(seed))


def _shuffled(keys, n, m, g):
    """m of the distinct pair keys lo * n + hi in random order, randomly oriented, as int32 [m, 2]."""
    keys = keys[torch.randperm(keys.shape[0], generator=g, device="cuda")[:m]]
    flip = torch.rand(m, generator=g, device="cuda") < 0.5
    u, v = keys // n, keys % n
    e = torch.stack([torch.where(flip, v, u), torch.where(flip, u, v)], 1)
    return e.to(torch.int32).contiguous()


def _collect(sample, n, m):
    """At least m distinct pair keys from batches of sampled endpoint pairs."""
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    while keys.shape[0] < m:
        u, v = sample(int((m - keys.shape[0]) * 1.25) + 1024)
        ok = u != v
        u, v = u[ok], v[ok]
        keys = torch.unique(torch.cat([keys, torch.minimum(u, v) * n + torch.maximum(u, v)]))
    return keys


def _rmat(case, g):
    n, scale, a, b = case["n"], case["scale"], case["a"], case["b"]

    def sample(count):
        u = torch.zeros(count, dtype=torch.int64, device="cuda")
        v = torch.zeros(count, dtype=torch.int64, device="cuda")
        for _ in range(scale):
            r = torch.rand(count, generator=g, device="cuda")
            bu = r >= a + b
            u = (u << 1) | bu
            v = (v << 1) | (((r >= a) & (r < a + b)) | (r >= a + 2 * b))
        ok = (u < n) & (v < n)
        return u[ok], v[ok]

    return _shuffled(_collect(sample, n, case["m"]), n, case["m"], g)


def _sizes(n, k, sigma, rng):
    """k community sizes of lognormal spread, at least 2 each, that sum to n."""
    w = rng.lognormal(0.0, sigma, size=k)
    s = np.floor(w / w.sum() * (n - 2 * k)).astype(np.int64) + 2
    s[np.argmax(s)] += n - s.sum()
    return s


def _planted(case, g, seed):
    """Edges and every node's community: a share `intra` of the edges joins two nodes of one community."""
    n, m, k = case["n"], case["m"], case["k"]
    sizes = _sizes(n, min(k, n // 4), 0.5, np.random.default_rng(seed))
    off = torch.from_numpy(np.concatenate([[0], np.cumsum(sizes)])).cuda()
    comm = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), torch.from_numpy(sizes).cuda())

    def sample(count):
        u = torch.randint(n, (count,), generator=g, device="cuda")
        c = comm[u]
        r = torch.rand(count, generator=g, device="cuda", dtype=torch.float64)
        inside = off[c] + (r * (off[c + 1] - off[c])).to(torch.int64)
        anywhere = torch.randint(n, (count,), generator=g, device="cuda")
        return u, torch.where(torch.rand(count, generator=g, device="cuda") < case["intra"], inside, anywhere)

    e = _shuffled(_collect(sample, n, m), n, m, g)
    perm = torch.randperm(n, generator=g, device="cuda")
    member = torch.empty(n, dtype=torch.int64, device="cuda")
    member[perm] = comm
    return perm[e.long()].to(torch.int32).contiguous(), member


def _edges(case, seed):
    g = _gen(seed)
    return _rmat(case, g) if case["graph"] == "rmat" else _planted(case, g, seed)[0]


def _i32(*shape):
    return torch.zeros(shape, dtype=torch.int32, device="cuda")


def _f32(*shape):
    return torch.zeros(shape, dtype=torch.float32, device="cuda")


def _i64(*shape):
    return torch.zeros(shape, dtype=torch.int64, device="cuda")


def _fa2_params(case):
    p = B.bgv_fa2_default_params()
    p.theta = case.get("theta", 1.2)
    p.leaf_cap = case.get("leaf_cap", 1)
    p.strong_gravity = case.get("strong", 0)
    return p


def _layout_params(case):
    p = B.bgv_layout_default_params()
    p.width = case["width"]
    p.threshold = case.get("threshold", 0)
    p.iterations = case["iterations"]
    return p


def _batch_nodes(case):
    """Node offsets of the batch's graphs: log-uniform sizes, the same for every seed."""
    r = np.random.default_rng(case["sizes"])
    sizes = np.exp(r.uniform(np.log(case["n_lo"]), np.log(case["n_hi"]), case["graphs"])).astype(np.int64)
    return np.concatenate([[0], np.cumsum(sizes)])


def _batch_graphs(case, seed):
    """Concatenated edge lists in local ids, grouped by graph, and the edge offsets."""
    rng, g = np.random.default_rng(seed), _gen(seed)
    node_off = _batch_nodes(case)
    G, N = case["graphs"], int(node_off[-1])
    parts = [_sizes(int(s), int(rng.integers(4, 65)), 0.5, rng) for s in np.diff(node_off)]
    sizes = np.concatenate(parts)
    coff = torch.from_numpy(np.concatenate([[0], np.cumsum(sizes)])).cuda()
    comm = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), torch.from_numpy(sizes).cuda())
    noff = torch.from_numpy(node_off).cuda()
    graph = torch.repeat_interleave(torch.arange(G, device="cuda"), noff[1:] - noff[:-1])
    m = int(N * case["degree"] / 2)
    u = torch.randint(N, (m,), generator=g, device="cuda")
    near = torch.rand(m, generator=g, device="cuda") < 0.8
    lo = torch.where(near, coff[comm[u]], noff[graph[u]])
    hi = torch.where(near, coff[comm[u] + 1], noff[graph[u] + 1])
    v = lo + (torch.rand(m, generator=g, device="cuda", dtype=torch.float64) * (hi - lo)).to(torch.int64)
    ok = u != v
    keys = torch.unique(torch.minimum(u[ok], v[ok]) * N + torch.maximum(u[ok], v[ok]))
    keys = keys[torch.randperm(keys.shape[0], generator=g, device="cuda")]
    perm = torch.argsort(graph * 2.0 + torch.rand(N, generator=g, device="cuda"))  # ids permuted inside each graph
    inv = torch.empty_like(perm)
    inv[perm] = torch.arange(N, device="cuda")
    gr = graph[keys // N]
    order = torch.argsort(gr, stable=True)
    keys, gr = keys[order], gr[order]
    e = torch.stack([inv[keys // N] - noff[gr], inv[keys % N] - noff[gr]], 1).to(torch.int32).contiguous()
    edge_off = np.concatenate([[0], np.cumsum(torch.bincount(gr, minlength=G).cpu().numpy())])
    return e, edge_off.astype(np.int64), node_off.astype(np.int32)


def _csr(e, n):
    """Symmetric CSR of a simple graph (ascending neighbours, unit weights) and mass = degree + 1."""
    e = e.long()
    key = torch.sort(torch.cat([e[:, 0] * n + e[:, 1], e[:, 1] * n + e[:, 0]])).values
    deg = torch.bincount(key // n, minlength=n)
    off = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), torch.cumsum(deg, 0)])
    adj = (key % n).to(torch.int32)
    return off.to(torch.int32), adj, torch.ones_like(adj), (deg + 1).to(torch.int32)


def _step_inputs(case, seed):
    """A layout part of the way through: communities apart, bodies spread around their centres, forces of the step
    before."""
    g, n = _gen(seed), case["n"]
    if case["graph"] == "rmat":
        e, member = _rmat(case, g), torch.randint(64, (n,), generator=g, device="cuda")
    else:
        e, member = _planted(case, g, seed)
    k = int(member.max()) + 1
    R = math.sqrt(n) * 4
    centre = torch.randn((k, 2), generator=g, device="cuda") * R
    pos = (centre[member] + torch.randn((n, 2), generator=g, device="cuda") * (R / 6)).contiguous()
    Fprev = (torch.randn((n, 2), generator=g, device="cuda") * 3).contiguous()
    return e, pos, Fprev


def prepare(case, seed):
    kind = case["kind"]
    if kind == "picture":
        g = _gen(seed)
        K, n = case["K"], case["n"]
        xy = (torch.randn((K, 2), generator=g, device="cuda") * math.sqrt(K) * 4).contiguous()
        mass = torch.exp(torch.randn(K, generator=g, device="cuda") * 1.5 + 1.0).to(torch.int32) + 1
        return {"kind": kind, "case": case, "xy": xy, "mass": mass, "radius": torch.sqrt(mass.float()),
                "node_map": torch.randint(K, (n,), generator=g, device="cuda", dtype=torch.int32),
                "group": torch.zeros(K, dtype=torch.uint8, device="cuda"),
                "colour": torch.zeros(n, dtype=torch.uint8, device="cuda"),
                "rgba": torch.zeros((case["H"], case["W"], 4), dtype=torch.uint8, device="cuda"),
                "ws_c": B.alloc_ws(B.bgv_colour_groups_ws_size(K)),
                "ws_r": B.alloc_ws(B.bgv_render_ws_size(case["W"], case["H"]))}
    if kind == "batch":
        e, edge_off, node_off = _batch_graphs(case, seed)
        G, N, p = case["graphs"], int(node_off[-1]), _layout_params(case)
        return {"kind": kind, "G": G, "e": e, "edge_off": edge_off, "node_off": node_off, "p": p, "node_map": _i32(N),
                "xy": _f32(N, 2), "radius": _f32(N),
                "ws": B.alloc_ws(B.bgv_layout_batched_ws_size(G, edge_off, node_off, p)),
                "stream": torch.cuda.Stream()}
    n, m = case["n"], case["m"]
    if kind == "step":
        e, pos, Fprev = _step_inputs(case, seed)
        off, adj, w, mass = _csr(e, n)
        return {"kind": kind, "n": n, "nnz": 2 * m, "off": off, "adj": adj, "w": w, "mass": mass, "pos": pos,
                "F": _f32(n, 2), "Fprev": Fprev, "speed": torch.ones(1, dtype=torch.float64, device="cuda"),
                "p": _fa2_params(case), "ws": B.alloc_ws(B.bgv_fa2_ws_size(n, 2 * m))}
    e = _edges(case, seed)
    if kind == "layout":
        p = _layout_params(case)
        s = {"kind": kind, "n": n, "m": m, "p": p, "host": case["host"], "stream": torch.cuda.Stream()}
        if case["host"]:
            h = torch.empty((m, 2), dtype=torch.int32, pin_memory=True)
            h.copy_(e)
            return {**s, "e": h, "node_map": torch.zeros(n, dtype=torch.int32, pin_memory=True),
                    "xy": torch.zeros((n, 2), dtype=torch.float32, pin_memory=True),
                    "radius": torch.zeros(n, dtype=torch.float32, pin_memory=True),
                    "ws": B.alloc_ws(B.bgv_layout_host_ws_size(m, n, p))}
        return {**s, "e": e, "node_map": _i32(n), "xy": _f32(n, 2), "radius": _f32(n),
                "ws": B.alloc_ws(B.bgv_layout_ws_size(m, n, p))}
    if kind == "csr":
        return {"kind": kind, "n": n, "m": m, "e": e, "off": _i32(n + 1), "adj": _i32(2 * m), "w": _i32(2 * m),
                "mass": _i32(n), "nnz": _i64(1), "ws": B.alloc_ws(B.bgv_graph_csr_ws_size(m, n))}
    if kind == "run":
        off, adj, w, mass = _csr(e, n)
        return {"kind": kind, "n": n, "nnz": 2 * m, "off": off, "adj": adj, "w": w, "mass": mass, "pos": _f32(n, 2),
                "F": _f32(n, 2), "Fprev": _f32(n, 2), "speed": torch.ones(1, dtype=torch.float64, device="cuda"),
                "p": _fa2_params(case), "iterations": case["iterations"], "stream": torch.cuda.Stream(),
                "ws": B.alloc_ws(B.bgv_fa2_ws_size(n, 2 * m))}
    rows, width = case["rows"], case["width"]
    s = {"kind": kind, "n": n, "m": m, "e": e, "rows": rows, "width": width, "sketch": _i32(rows, width),
         "deg": _i32(n), "case": case}
    ws = B.alloc_ws(B.bgv_sketch_degrees_ws_size(m, n, rows, width))
    if kind == "sketch":
        return {**s, "ws": ws}
    # the stages after the sketch start from its degrees, as in a user's chain of calls
    B.bgv_sketch_degrees(e, m, n, rows, width, 1, s["sketch"], s["deg"], ws)
    if kind == "communities":
        return {**s, "labels": _i32(n), "deg_out": _i32(n), "ws": B.alloc_ws(B.bgv_communities_ex_ws_size(m, n))}
    labels = _i32(n)
    B.bgv_communities(e, m, n, s["deg"], 3, 0, 2, 0, labels, None, B.alloc_ws(B.bgv_communities_ws_size(m, n)))
    opt = case["optional"]
    return {**s, "labels": labels, "node_map": _i32(n), "K": _i64(1), "Es": _i64(1), "ssrc": _i32(m), "sdst": _i32(m),
            "sw": _i32(m), "mass": _i32(n), "off": _i32(n + 1), "adj": _i32(2 * m), "w": _i32(2 * m),
            "vol": _i64(n) if opt else None, "count": _i32(n) if opt else None,
            "comm_label": _i32(n) if opt else None, "ws": B.alloc_ws(B.bgv_supergraph_ws_size(m, n, rows, width))}


def run(s):
    kind = s["kind"]
    if kind == "layout":
        f = B.bgv_layout_host if s["host"] else B.bgv_layout
        s["stream"].wait_stream(torch.cuda.current_stream())
        K, Es = f(s["e"], s["m"], s["n"], s["p"], s["node_map"], s["xy"], s["radius"], s["ws"], stream=s["stream"])
        return {"K": K, "Es": Es, "node_map": s["node_map"], "xy": s["xy"], "radius": s["radius"]}
    if kind == "batch":
        s["stream"].wait_stream(torch.cuda.current_stream())
        K_off, Es_off = B.bgv_layout_batched(s["e"], s["G"], s["edge_off"], s["node_off"], s["p"], s["node_map"],
                                             s["xy"], s["radius"], s["ws"], stream=s["stream"])
        return {"K_off": K_off, "Es_off": Es_off, "node_map": s["node_map"], "xy": s["xy"], "radius": s["radius"]}
    if kind == "sketch":
        B.bgv_sketch_degrees(s["e"], s["m"], s["n"], s["rows"], s["width"], 1, s["sketch"], s["deg"], s["ws"])
        return {"sketch": s["sketch"], "deg": s["deg"]}
    if kind == "communities":
        c = s["case"]
        D = B.bgv_communities_ex(s["e"], s["m"], s["n"], s["deg"], c["passes"], c["threshold"], 2, c["tie_mode"],
                                 c["mode"], c["jumps"], s["labels"], s["deg_out"], s["ws"])
        return {"labels": s["labels"], "deg": s["deg_out"], "threshold": D}
    if kind == "supergraph":
        B.bgv_supergraph(s["e"], s["m"], s["n"], s["labels"], s["deg"], s["rows"], s["width"], 1, s["node_map"],
                         s["K"], s["ssrc"], s["sdst"], s["sw"], s["Es"], s["mass"], s["off"], s["adj"], s["w"],
                         s["vol"], s["count"], s["comm_label"], s["ws"])
        out = {k: s[k] for k in ("K", "Es", "node_map", "ssrc", "sdst", "sw", "mass", "off", "adj", "w")}
        if s["vol"] is not None:
            out.update(vol=s["vol"], count=s["count"], comm_label=s["comm_label"])
        return out
    if kind == "csr":
        B.bgv_graph_csr(s["e"], s["m"], s["n"], s["off"], s["adj"], s["w"], s["mass"], s["nnz"], s["ws"])
        return {"off": s["off"], "adj": s["adj"], "w": s["w"], "mass": s["mass"], "nnz": s["nnz"]}
    if kind == "run":
        st = s["stream"]
        st.wait_stream(torch.cuda.current_stream())
        B.bgv_fa2_init(s["n"], s["p"], s["pos"], s["Fprev"], s["speed"], stream=st)
        B.bgv_fa2_run(s["n"], s["nnz"], s["off"], s["adj"], s["w"], s["mass"], s["p"], s["iterations"], True,
                      s["pos"], s["F"], s["Fprev"], s["speed"], s["ws"], stream=st)
        torch.cuda.current_stream().wait_stream(st)
        return {"pos": s["pos"], "F": s["F"], "Fprev": s["Fprev"], "speed": s["speed"]}
    if kind == "step":
        B.bgv_fa2_step(s["n"], s["nnz"], s["off"], s["adj"], s["w"], s["mass"], s["p"], s["pos"], s["F"], s["Fprev"],
                       s["speed"], s["ws"])
        return {"pos": s["pos"], "F": s["F"], "Fprev": s["Fprev"], "speed": s["speed"]}
    c = s["case"]
    B.bgv_colour_groups(c["K"], s["mass"], s["group"], s["ws_c"], c["n"], s["node_map"], s["colour"])
    B.bgv_render(c["K"], s["xy"], s["radius"], s["group"], c["W"], c["H"], s["rgba"], s["ws_r"])
    return {"group": s["group"], "colour": s["colour"], "rgba": s["rgba"]}


# -------------------------------------------------------------------- work
def _fa2_work(K, nnz, iterations):
    """An iteration reads every CSR entry (id, weight) and the bodies' mass, position and previous force, and writes
    position and force; about 60 repulsion terms a body at theta 1.2 (12 operations each), 6 operations an entry."""
    return iterations * (8.0 * nnz + 36.0 * K), iterations * (60 * 12.0 * K + 6.0 * nnz)


def work(case):
    kind = case["kind"]
    if kind == "picture":
        K, n, px = case["K"], case["n"], case["W"] * case["H"]
        return {"bytes": 17.0 * K + 5.0 * n + 4.0 * px, "flops": 10.0 * K}
    if kind == "batch":
        n = int(_batch_nodes(case)[-1])
        m = int(n * case["degree"] / 2)
        b, f = _fa2_work(n, 2 * m, case["iterations"])
        return {"bytes": 8.0 * m + 16.0 * n + b, "flops": f}
    n, m = case["n"], case["m"]
    if kind == "layout":  # most nodes stay communities of their own, most edges superedges
        b, f = _fa2_work(n, 2 * m, case["iterations"])
        return {"bytes": 8.0 * m + 16.0 * n + b, "flops": f}
    if kind in ("run", "step"):
        b, f = _fa2_work(n, 2 * m, case.get("iterations", 1))
        return {"bytes": b, "flops": f}
    if kind == "csr":
        return {"bytes": 8.0 * m + 16.0 * m + 8.0 * n, "flops": 0.0}
    if kind == "sketch":
        return {"bytes": 8.0 * m + 4.0 * n + 4.0 * case["rows"] * case["width"], "flops": 0.0}
    if kind == "communities":
        return {"bytes": 8.0 * m + 12.0 * n, "flops": 0.0}
    return {"bytes": 8.0 * m + 8.0 * n + 28.0 * m + 12.0 * n, "flops": 0.0}


# ------------------------------------------------------------------- exact
def _spread(v):
    x = v.astype(np.uint64)
    for s, mask in ((16, 0x0000FFFF0000FFFF), (8, 0x00FF00FF00FF00FF), (4, 0x0F0F0F0F0F0F0F0F),
                    (2, 0x3333333333333333), (1, 0x5555555555555555)):
        x = (x | (x << np.uint64(s))) & np.uint64(mask)
    return x


def _repulsion(pos, mass, theta, leaf_cap, L, kr):
    """Barnes-Hut repulsion as the method defines it, level by level over all (body, cell) pairs: the opening test in
    FP32 on centres from exact integer moments, the forces in FP64."""
    f32 = np.float32
    K = pos.shape[0]
    lo = pos.min(0)
    side = f32(max(pos.max(0) - lo)) * f32(1.00000095367431640625)
    U = (((pos - lo) / side) * f32(4294967296.0)).astype(np.uint64)
    q = U >> np.uint64(32 - L)
    key = (_spread(q[:, 0]) << np.uint64(1)) | _spread(q[:, 1])
    order = np.argsort(key, kind="stable")
    key, p, m, U = key[order], pos[order], mass[order].astype(np.int64), U[order].astype(np.int64)
    P = np.zeros((K + 1, 3), np.int64)  # masses and sizes here keep the sums below 2^63
    P[1:] = np.cumsum(np.stack([m, m * U[:, 0], m * U[:, 1]], 1), 0)
    p64, m64 = p.astype(np.float64), m.astype(np.float64)
    F = np.zeros((K, 2))
    theta2 = f32(theta) * f32(theta)

    def firsts(lev):
        pre = key >> np.uint64(2 * (L - lev))
        return np.concatenate([[0], np.nonzero(pre[1:] != pre[:-1])[0] + 1, [K]])

    def add(s, d, w):
        d2 = (d * d).sum(1)
        f = np.where(d2 > 0, kr * m64[s] * w / np.where(d2 > 0, d2, 1.0), 0.0)
        for ax in (0, 1):
            F[:, ax] += np.bincount(s, f * d[:, ax], K)

    def ranges(s, a, b):
        cnt = b - a
        at = np.repeat(a - np.concatenate([[0], np.cumsum(cnt)[:-1]]), cnt) + np.arange(cnt.sum())
        return np.repeat(s, cnt), at

    here = firsts(0)
    s, c = np.arange(K), np.zeros(K, np.int64)
    for lev in range(L + 1):
        a, b = here[c], here[c + 1]
        inside = (a <= s) & (s < b)
        leaf = (b - a <= leaf_cap) | (lev == L)
        ls, lt = ranges(s[leaf], a[leaf], b[leaf])
        keep = ls != lt
        add(ls[keep], p64[ls[keep]] - p64[lt[keep]], m64[lt[keep]])
        s, c, a, b, inside = s[~leaf], c[~leaf], a[~leaf], b[~leaf], inside[~leaf]
        if not s.size:
            break
        mom = P[here[1:]] - P[here[:-1]]
        cen = (mom[:, 1:] // mom[:, :1]).astype(f32) * f32(2.3283064365386963e-10)
        cen = lo + side * cen
        d = p[s] - cen[c]
        sl = side * f32(2.0 ** -lev)
        take = ~inside & (sl * sl < theta2 * (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]))
        add(s[take], p64[s[take]] - cen[c[take]].astype(np.float64), mom[c[take], 0].astype(np.float64))
        s, a, b = s[~take], a[~take], b[~take]
        here = firsts(lev + 1)
        s, c = ranges(s, np.searchsorted(here, a), np.searchsorted(here, b))
    out = np.zeros((K, 2))
    out[order] = F
    return out


def exact(case, seed):
    """One ForceAtlas2 step in 64 bits.  The other kinds give whole numbers and bytes, or runs of hundreds of steps,
    which are chaotic."""
    if case["kind"] != "step" or case["n"] > 100_000 or case["m"] > 1_000_000:
        return None
    e, pos, Fprev = (t.cpu().numpy() for t in _step_inputs(case, seed))
    n = case["n"]
    deg = np.bincount(e.reshape(-1), minlength=n)
    mass, p, Fp = deg + 1, pos.astype(np.float64), Fprev.astype(np.float64)
    F = _repulsion(pos, mass, case["theta"], case["leaf_cap"], 24, 2.0)
    d = p[e[:, 1]] - p[e[:, 0]]  # unit weights
    r = np.linalg.norm(p, axis=1)
    for ax in (0, 1):
        F[:, ax] += np.bincount(e[:, 0], d[:, ax], n) - np.bincount(e[:, 1], d[:, ax], n)
        F[:, ax] -= mass * p[:, ax] / (1.0 if case["strong"] else np.where(r > 0, r, 1.0))
    swing = np.linalg.norm(F - Fp, axis=1)
    S, T = (mass * swing).sum(), (mass * np.linalg.norm(F + Fp, axis=1) / 2).sum()
    speed = 1.0 + min(T / S - 1.0, 0.5)
    norm = np.linalg.norm(F, axis=1)
    s = 0.1 * speed / (1.0 + speed * np.sqrt(swing))
    s = np.where((norm > 0) & (s * norm > 10.0), 10.0 / np.where(norm > 0, norm, 1.0), s)
    return {"pos": p + s[:, None] * F, "F": F, "Fprev": F, "speed": np.array([speed])}

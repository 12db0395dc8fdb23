"""Measured workloads of the push-pull BFS library, through its Python binding and C ABI.

listed() gives the workloads, draw() more of the same ranges.  Inputs are drawn on the GPU from
the seed: RMAT graphs (a, b, c, d = 0.57, 0.19, 0.19, 0.05, vertex ids relabelled), 4-neighbour
grids with 1 % of the edges deleted, sources among the vertices that have an edge, random frontier
and mask vectors, and edge weights.

Depths, distances, CSR arrays and matvec results are returned whole.  Parents are computed where
the case says so, as a Graph500-style user asks for them, but not returned: any in-neighbour one
level up is a valid parent and the one recorded differs from run to run.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1804_03327_gb300 import gbx

DEV = "cuda"


def listed():
    return [
        # one BFS of a small graph: launch and per-level latency
        {"name": "bfs_rmat10", "kind": "bfs", "graph": "rmat", "n": 1 << 10, "ef": 16, "directed": False,
         "sources": 1, "parent": True, "alpha": 0.01, "beta": 0.01},
        # the headline workload: direction-optimised BFS of RMAT-22, depth and parent, source after
        # source, with thresholds as gbx_autotune returns them for this graph
        {"name": "bfs_rmat22", "kind": "bfs", "graph": "rmat", "n": 1 << 22, "ef": 16, "directed": False,
         "sources": 8, "parent": True, "alpha": 0.001, "beta": 0.0},
        # a road-like graph: thousands of small levels, default descriptor
        {"name": "bfs_grid2048", "kind": "bfs", "graph": "grid", "width": 2048, "height": 2048, "directed": False,
         "sources": 1, "parent": True, "alpha": 0.01, "beta": 0.01},
        # a batch of 64 sources as one word of lanes (threshold as tuned), int32 depths
        {"name": "batch_rmat21_s64", "kind": "batch", "graph": "rmat", "n": 1 << 21, "ef": 16, "directed": False,
         "lanes": 64, "depth16": False, "alpha": 0.2},
        # a wide batch whose last lane word is ragged, int16 depths, default threshold
        {"name": "batch_rmat20_s1000", "kind": "batch", "graph": "rmat", "n": 1 << 20, "ef": 16, "directed": False,
         "lanes": 1000, "depth16": True, "alpha": 0.01},
        # queries over several resident graphs through the continuous-batching server
        {"name": "serve_mix", "kind": "serve", "scale_lo": 16, "scale_hi": 20, "side": 1024, "queries": 256,
         "slots": 4},
        # shortest paths on a skewed graph, integer weights 1..64, default descriptor
        {"name": "sssp_rmat22", "kind": "sssp", "graph": "rmat", "n": 1 << 22, "ef": 16, "directed": False,
         "integer": True, "alpha": 0.01, "beta": 0.01},
        # shortest paths on a road-like graph of odd sides with real lengths
        {"name": "sssp_grid777", "kind": "sssp", "graph": "grid", "width": 1001, "height": 777, "directed": False,
         "integer": False, "alpha": 0.01, "beta": 0.01},
        # one early BFS step as a user's own loop issues it: tiny sparse frontier, complemented
        # visited mask, sparse result
        {"name": "mxv_push_rmat20", "kind": "mxv", "graph": "rmat", "n": 1 << 20, "ef": 16, "directed": False,
         "frontier": 0.0001, "visited": 0.01, "sparse": True, "accum": False, "direction": 0},
        # one heavy BFS step: byte vectors, a fifth of the vertices in the frontier, half visited
        {"name": "mxv_pull_rmat22", "kind": "mxv", "graph": "rmat", "n": 1 << 22, "ef": 16, "directed": False,
         "frontier": 0.2, "visited": 0.5, "sparse": False, "accum": False, "direction": 0},
        # a (min, +) matvec on a directed graph of odd size, accumulating
        {"name": "minplus_directed", "kind": "minplus", "graph": "rmat", "n": 700001, "ef": 16, "directed": True,
         "frontier": 0.3, "visited": -1.0, "accum": True, "direction": 0},
        # edge list on the device -> graph with weights, taken out again as CSR
        {"name": "build_rmat20", "kind": "build", "graph": "rmat", "n": 1 << 20, "ef": 16, "directed": False,
         "weights": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_rmat(rng, lo, hi):
    return {"graph": "rmat", "n": _log_int(rng, lo, hi), "ef": rng.choice([4, 8, 16, 24]),
            "directed": rng.random() < 0.3}


def _draw_grid(rng, lo, hi):
    return {"graph": "grid", "width": _log_int(rng, lo, hi), "height": _log_int(rng, lo, hi), "directed": False}


def draw(rng):
    kind = rng.choice(["bfs", "bfs", "batch", "sssp", "mxv", "mxv", "minplus", "build", "serve"])
    c = {"kind": kind}
    if kind == "bfs":
        c.update(_draw_rmat(rng, 1000, 2500000) if rng.random() < 0.6 else _draw_grid(rng, 30, 1500))
        alpha, beta = rng.choice([(0.01, 0.01), (0.001, 0.0), (0.01, 0.0)])
        c.update(sources=rng.randint(1, 4) if c["graph"] == "rmat" else 1, parent=rng.random() < 0.7, alpha=alpha,
                 beta=beta)
    elif kind == "batch":
        if rng.random() < 0.7:
            c.update(_draw_rmat(rng, 1000, 1000000), lanes=_log_int(rng, 2, 700), alpha=rng.choice([0.01, 0.05, 0.2]))
        else:
            c.update(_draw_grid(rng, 30, 700), lanes=_log_int(rng, 2, 64), alpha=1e30)
        c["depth16"] = rng.random() < 0.5
    elif kind == "sssp":
        c.update(_draw_rmat(rng, 1000, 2500000) if rng.random() < 0.6 else _draw_grid(rng, 30, 700))
        alpha, beta = rng.choice([(0.01, 0.01), (0.2, 0.3)])
        c.update(integer=rng.random() < 0.5, alpha=alpha, beta=beta)
    elif kind in ("mxv", "minplus"):
        c.update(_draw_rmat(rng, 1000, 2500000) if rng.random() < 0.7 else _draw_grid(rng, 30, 1500))
        c.update(frontier=math.exp(rng.uniform(math.log(1e-5), math.log(0.5))),
                 visited=rng.choice([-1.0, 0.01, 0.3, 0.7, 0.99]), accum=rng.random() < 0.3,
                 direction=rng.choice([0, 0, 1, 2]))
        if kind == "mxv":
            c["sparse"] = rng.random() < 0.5
    elif kind == "build":
        c.update(_draw_rmat(rng, 1000, 600000) if rng.random() < 0.7 else _draw_grid(rng, 30, 1500))
        c["weights"] = rng.random() < 0.5
    else:
        lo = rng.randint(10, 16)
        c.update(scale_lo=lo, scale_hi=rng.randint(lo, 19), side=_log_int(rng, 30, 600), queries=_log_int(rng, 4, 300),
                 slots=rng.choice([1, 2, 4]))
    return c


# ---------------------------------------------------------------- inputs


def _rmat(n, ef, gen):
    """ef * n directed RMAT samples on [0, n): ids of the next power of two, relabelled, scaled down to n."""
    scale = max(1, (n - 1).bit_length())
    m = ef * n
    src = torch.zeros(m, dtype=torch.int32, device=DEV)
    dst = torch.zeros(m, dtype=torch.int32, device=DEV)
    for _ in range(scale):
        r = torch.rand(m, generator=gen, device=DEV)
        src.mul_(2).add_(r >= 0.76)
        dst.mul_(2).add_(((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    perm = (torch.randperm(1 << scale, generator=gen, device=DEV) * n) >> scale
    perm = perm.to(torch.int32)
    return perm[src], perm[dst]


def _grid(width, height, gen):
    """The edges of a 4-neighbour grid (each once), 1 % of them deleted."""
    v = torch.arange(width * height, dtype=torch.int32, device=DEV).view(height, width)
    src = torch.cat([v[:, :-1].reshape(-1), v[:-1].reshape(-1)])
    dst = torch.cat([v[:, 1:].reshape(-1), v[1:].reshape(-1)])
    keep = torch.rand(src.numel(), generator=gen, device=DEV) >= 0.01
    return src[keep].contiguous(), dst[keep].contiguous()


def _edges(case, gen):
    if case["graph"] == "rmat":
        return (case["n"], *_rmat(case["n"], case["ef"], gen))
    return (case["width"] * case["height"], *_grid(case["width"], case["height"], gen))


def _weights(case, m, gen):
    if case.get("integer", True):
        return torch.randint(1, 65, (m,), generator=gen, device=DEV).to(torch.float32)
    return torch.rand(m, generator=gen, device=DEV) * 0.9 + 0.1


def _sources(n, src, dst, k, gen):
    """k vertices that have an out-edge to another vertex (repeated when there are fewer)."""
    has = torch.zeros(n, dtype=torch.bool, device=DEV)
    has[src[src != dst].long()] = True
    ids = torch.nonzero(has).view(-1)
    if ids.numel() == 0:
        return np.zeros(k, dtype=np.int32)
    return ids[torch.randint(0, ids.numel(), (k,), generator=gen, device=DEV)].cpu().numpy().astype(np.int32)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _build(case, n, src, dst):
    return gbx.graph_build(n, src, dst, symmetrize=not case.get("directed", False))


def _set(n, density, gen):
    return (torch.rand(n, generator=gen, device=DEV) < density).to(torch.uint8)


def _vectors(case, n, gen):
    """u, mask and w of a Boolean matvec: (gbx views, the tensors behind them)."""
    u, m = _set(n, case["frontier"], gen), _set(n, max(0.0, case["visited"]), gen)
    if not case["sparse"]:
        w = _set(n, 0.001, gen) if case["accum"] else torch.zeros(n, dtype=torch.uint8, device=DEV)
        mask = gbx.dense(m) if case["visited"] >= 0 else None
        return gbx.dense(u), mask, gbx.dense(w), (u, m, w, None)
    ids = torch.full((n,), -1, dtype=torch.int32, device=DEV)
    nnz = torch.zeros(1, dtype=torch.int32, device=DEV)
    if case["accum"]:
        old = torch.nonzero(_set(n, 0.001, gen)).view(-1).to(torch.int32)
        ids[: old.numel()] = old
        nnz.fill_(old.numel())
    ul = torch.nonzero(u).view(-1).to(torch.int32)
    uc = torch.tensor([ul.numel()], dtype=torch.int32, device=DEV)
    if ul.numel() == 0:
        ul = torch.zeros(1, dtype=torch.int32, device=DEV)
    mask = gbx.dense(m) if case["visited"] >= 0 else None
    return gbx.sparse(ul, uc, n), mask, gbx.sparse(ids, nnz, n), (ul, uc, m, ids, nnz)


def _minplus_vectors(case, n, gen):
    u = torch.rand(n, generator=gen, device=DEV) * 100.0
    u[torch.rand(n, generator=gen, device=DEV) >= case["frontier"]] = float("inf")
    m = _set(n, max(0.0, case["visited"]), gen)
    w = torch.rand(n, generator=gen, device=DEV) * 40.0 + 1.0
    return u, m, w


def prepare(case, seed):
    gen = _gen(seed)
    kind = case["kind"]
    if kind == "serve":
        return _prepare_serve(case, gen)
    n, src, dst = _edges(case, gen)
    st = {"kind": kind, "n": n}
    if kind == "build":
        st.update(src=src, dst=dst, w=_weights(case, src.numel(), gen) if case["weights"] else None,
                  directed=case["directed"], out={})
        cap = src.numel() * (1 if case["directed"] else 2)  # entries before duplicates are removed
        for t in (0, 1) if case["directed"] else (0,):
            st["out"][f"ptr{t}"] = torch.empty(n + 1, dtype=torch.int32, device=DEV)
            st["out"][f"col{t}"] = torch.full((cap,), -1, dtype=torch.int32, device=DEV)
            if case["weights"]:
                st["out"][f"val{t}"] = torch.full((cap,), float("inf"), dtype=torch.float32, device=DEV)
        return st
    g = st["g"] = _build(case, n, src, dst)
    if kind == "bfs":
        k = case["sources"]
        st.update(sources=[int(s) for s in _sources(n, src, dst, k, gen)],
                  depth=torch.empty((k, n), dtype=torch.int32, device=DEV),
                  parent=torch.empty((k, n), dtype=torch.int32, device=DEV) if case["parent"] else None,
                  desc=gbx.desc_init(alpha=case["alpha"], beta=case["beta"]))
    elif kind == "batch":
        dt = torch.int16 if case["depth16"] else torch.int32
        st.update(sources=_sources(n, src, dst, case["lanes"], gen),
                  depth=torch.empty((case["lanes"], n), dtype=dt, device=DEV), desc=gbx.desc_init(alpha=case["alpha"]))
    elif kind == "sssp":
        gbx.graph_set_weights(g, src, dst, _weights(case, src.numel(), gen))
        st.update(source=int(_sources(n, src, dst, 1, gen)[0]), dist=torch.empty(n, dtype=torch.float32, device=DEV),
                  desc=gbx.desc_init(alpha=case["alpha"], beta=case["beta"]))
    elif kind == "mxv":
        u, mask, w, held = _vectors(case, n, gen)
        st.update(u=u, mask=mask, w=w, held=held,
                  desc=gbx.desc_init(mask_complement=1 if mask is not None else 0, accum=int(case["accum"]),
                                     direction=case["direction"]))
    else:
        gbx.graph_set_weights(g, src, dst, _weights(case, src.numel(), gen))
        u, m, w = _minplus_vectors(case, n, gen)
        mask = gbx.dense(m) if case["visited"] >= 0 else None
        st.update(u=gbx.dense_f32(u), mask=mask, w=gbx.dense_f32(w), held=(u, m, w),
                  desc=gbx.desc_init(mask_complement=1 if mask is not None else 0, accum=int(case["accum"]),
                                     direction=case["direction"]))
    return st


def _prepare_serve(case, gen):
    """RMAT graphs of the even scales from scale_lo to scale_hi and a square grid, resident in one server."""
    graphs, rows, queries = [], [], []
    specs = [{"graph": "rmat", "n": 1 << s, "ef": 16} for s in range(case["scale_lo"], case["scale_hi"] + 1, 2)]
    specs.append({"graph": "grid", "width": case["side"], "height": case["side"]})
    server = gbx.Server(slots=case["slots"], depth_type=gbx.DEPTH_I16)
    per = [case["queries"] // len(specs) + (i < case["queries"] % len(specs)) for i in range(len(specs))]
    for spec, k in zip(specs, per):
        n, src, dst = _edges(spec, gen)
        g = gbx.graph_build(n, src, dst)
        gid = server.add_graph(g)
        server.set_graph_desc(gid, gbx.desc_init(alpha=0.5 if spec["graph"] == "rmat" else 1e30))
        out = torch.empty((k, n), dtype=torch.int16, device=DEV)
        queries.append([(gid, int(s), out[i]) for i, s in enumerate(_sources(n, src, dst, k, gen))])
        graphs.append(g)
        rows.append(out)
    # arrivals alternate between the graphs
    mixed = [q[i] for i in range(max(per)) for q in queries if i < len(q)]
    torch.cuda.synchronize()
    return {"kind": "serve", "server": server, "graphs": graphs, "rows": rows, "queries": mixed}


# ---------------------------------------------------------------- one pass


def run(state):
    kind = state["kind"]
    if kind == "bfs":
        for i, s in enumerate(state["sources"]):
            gbx.bfs(state["g"], s, state["depth"][i], state["parent"][i] if state["parent"] is not None else None,
                    state["desc"])
        return state["depth"]
    if kind == "batch":
        gbx.bfs_batch(state["g"], state["sources"], state["depth"], state["desc"])
        return state["depth"]
    if kind == "serve":
        server, left = state["server"], len(state["queries"])
        for tag, (gid, s, out) in enumerate(state["queries"]):
            server.submit(gid, s, out, tag)
        while left:
            for c in server.poll():
                if c.status:
                    raise RuntimeError(f"query {c.tag}: status {c.status}")
                left -= 1
        return state["rows"]
    if kind == "sssp":
        gbx.sssp(state["g"], state["source"], state["dist"], state["desc"])
        return state["dist"]
    if kind in ("mxv", "minplus"):
        gbx.mxv(state["w"], state["mask"], gbx.LOR_LAND if kind == "mxv" else gbx.MIN_PLUS_F32, state["g"], state["u"],
                state["desc"])
        held = state["held"]
        return {"ids": held[3], "nnz": held[4]} if len(held) == 5 else held[2]
    return _run_build(state)


def _run_build(state):
    g = gbx.graph_build(state["n"], state["src"], state["dst"], symmetrize=not state["directed"])
    out, lib = state["out"], gbx.load()
    if state["w"] is not None:
        gbx.graph_set_weights(g, state["src"], state["dst"], state["w"])
    for t in (0, 1) if state["directed"] else (0,):
        if lib.gbx_graph_copy_csr(g.handle, t, out[f"ptr{t}"].data_ptr(), out[f"col{t}"].data_ptr()):
            raise RuntimeError("gbx_graph_copy_csr failed")
        if state["w"] is not None and lib.gbx_graph_copy_weights(g.handle, t, out[f"val{t}"].data_ptr()):
            raise RuntimeError("gbx_graph_copy_weights failed")
    g.free()
    return out


# ---------------------------------------------------------------- what a pass cannot do without


def _shape(case):
    """(n, stored entries of A), the latter without the few duplicates."""
    if case["graph"] == "rmat":
        return case["n"], case["ef"] * case["n"] * (1 if case["directed"] else 2)
    n = case["width"] * case["height"]
    return n, 4 * n


def work(case):
    kind = case["kind"]
    if kind == "serve":
        sizes = [1 << s for s in range(case["scale_lo"], case["scale_hi"] + 1, 2)] + [case["side"] ** 2]
        per = case["queries"] / len(sizes)
        # every query's int16 row out; every vertex's entry of the adjacency at least once a graph
        return {"bytes": sum(2 * n * per + 8 * n for n in sizes), "flops": 0}
    n, nnz = _shape(case)
    if kind == "bfs":
        # the outputs, and one in-edge of every vertex with its place in the rows
        return {"bytes": case["sources"] * n * (8 + 4 + (4 if case["parent"] else 0)), "flops": 0}
    if kind == "batch":
        # the rows of depths, and the adjacency once
        return {"bytes": case["lanes"] * n * (2 if case["depth16"] else 4) + 4 * n + 4 * nnz, "flops": 0}
    if kind == "sssp":
        # every edge relaxed once: neighbour and weight, and the distances out
        return {"bytes": 4 * n + 8 * nnz + 4 * n, "flops": nnz}
    if kind == "mxv":
        # the smaller of the frontier's rows and one entry of each computed row, and the vectors
        rows = n * (1.0 - max(0.0, case["visited"]))
        reach = min(case["frontier"] * nnz, rows)
        vec = (4 * case["frontier"] * n if case["sparse"] else 2 * n) + (n if case["visited"] >= 0 else 0)
        return {"bytes": 4 * reach + vec, "flops": 0}
    if kind == "minplus":
        rows = 1.0 - max(0.0, case["visited"])
        return {"bytes": 8 * nnz * min(rows, case["frontier"]) + 12 * n, "flops": nnz * min(rows, case["frontier"])}
    m = nnz if case["directed"] or case["graph"] == "grid" else nnz / 2
    each = 2 if case["directed"] else 1
    val = 4 if case["weights"] else 0
    return {"bytes": (8 + val) * m + each * (4 * n + (4 + val) * nnz), "flops": 0}


# ---------------------------------------------------------------- the same in 64 bits


def _pairs(case, src, dst, w):
    """The directed entries (row, col, value) of A, duplicates left in, self-loops dropped."""
    keep = src != dst
    src, dst, w = src[keep], dst[keep], w[keep].double()
    if case.get("directed", False):
        return src.long(), dst.long(), w
    return torch.cat([src, dst]).long(), torch.cat([dst, src]).long(), torch.cat([w, w])


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("sssp", "minplus", "build") or (kind == "build" and not case["weights"]):
        return None
    gen = _gen(seed)
    n, src, dst = _edges(case, gen)
    w = _weights(case, src.numel(), gen)
    if kind == "build":
        return _exact_build(case, n, src, dst, w)
    rows, cols, val = _pairs(case, src, dst, w)
    inf = float("inf")
    if kind == "minplus":
        u, m, old = _minplus_vectors(case, n, gen)
        t = torch.full((n,), inf, dtype=torch.float64, device=DEV)
        t.scatter_reduce_(0, cols, u.double()[rows] + val, "amin")
        ok = (m == 0) if case["visited"] >= 0 else torch.ones(n, dtype=torch.bool, device=DEV)
        base = old.double() if case["accum"] else torch.full((n,), inf, dtype=torch.float64, device=DEV)
        return torch.where(ok, torch.minimum(base, t), base)
    s = int(_sources(n, src, dst, 1, gen)[0])
    d = torch.full((n,), inf, dtype=torch.float64, device=DEV)
    d[s] = 0.0
    while True:
        was = d.clone()
        for _ in range(4):
            d.scatter_reduce_(0, cols, d[rows] + val, "amin")
        if torch.equal(was, d):
            return d


def _exact_build(case, n, src, dst, w):
    rows, cols, val = _pairs(case, src, dst, w)
    out = {}
    for t in (0, 1) if case["directed"] else (0,):
        key, inv = torch.unique((cols * n + rows) if t else (rows * n + cols), return_inverse=True)
        cap = src.numel() * (1 if case["directed"] else 2)
        v = torch.full((cap,), float("inf"), dtype=torch.float64, device=DEV)
        out[f"val{t}"] = v.scatter_reduce_(0, inv, val, "amin")
        out[f"ptr{t}"] = out[f"col{t}"] = None
    return out

"""The work that users of grx have it do, as cases that can be timed and compared.

A case is one call (one pass) of a public entry point on a loaded graph: what
a program does again and again once its graph is on the GPU.  The graphs are
the workloads of the benchmark and the serving loop: seeded R-MAT graphs
(scale 16 to 26, edge factor 16 unless drawn otherwise) and weighted grids of
high diameter.  Drawn cases add odd vertex counts (an R-MAT graph cut down to
its first nv vertices, grids of any width and height), other edge factors,
32- and 64-bit row offsets, and the batched forms of every size.

``prepare`` builds and loads the graph, picks the sources and fills in the
options; the traversal workspace is made by the first pass, as it is for a
user.  ``run`` makes one call and returns its whole output.
"""
import random

import torch

from paper_1504_04804_gb300 import grx


def _rmat(scale, ef=16, nv=0):
    return {"graph": "rmat", "scale": scale, "ef": ef, "nv": nv or 1 << scale, "offsets64": scale >= 26}


def _grid(width, height):
    return {"graph": "grid", "width": width, "height": height, "nv": width * height, "offsets64": False}


def listed():
    return [
        # the smallest call: one plain (push) BFS on a graph that fits in L2,
        # where launches, barriers and dependent round trips are the time
        dict(_rmat(16), name="bfs_rmat16", op="bfs", direction=grx.GRX_DIR_PUSH),
        # the headline traversal: direction-optimising BFS of one source
        dict(_rmat(22), name="dobfs_rmat22", op="bfs", alpha=1e-4, beta=0.01),
        # the same on the largest graph, with 64-bit row offsets
        dict(_rmat(26), name="dobfs_rmat26", op="bfs", alpha=1e-5, beta=0.01, push_bitmap=0.03125),
        # thousands of levels of small frontiers: routing on a road-like graph
        dict(_grid(4096, 4096), name="bfs_grid4096", op="bfs", direction=grx.GRX_DIR_PUSH),
        # weighted distances of one source on a social-network-like graph
        dict(_rmat(22), name="sssp_rmat22", op="sssp", wmax=64),
        # weighted distances on a road-like graph, in near-far bands
        dict(_grid(4096, 4096), name="sssp_grid4096", op="sssp", wmax=1000, sssp_delta=128132),
        # component labels of a whole graph
        dict(_rmat(22), name="cc_rmat22", op="cc"),
        # a whole ranking, on a graph whose ranks fit in L2 and on one whose do not
        dict(_rmat(22), name="pagerank_rmat22", op="pagerank", iters=20),
        dict(_rmat(26), name="pagerank_rmat26", op="pagerank", iters=20),
        # a full batch of hop-distance queries on the largest served graph
        dict(_rmat(24), name="bfs64_rmat24", op="bfs_multi", n=64, alpha=0.05, beta=1.0),
        # a part-filled batch of weighted queries on a served graph of middle size
        dict(_rmat(20), name="sssp16_rmat20", op="sssp_multi", wmax=64, n=16),
        # betweenness from a few sampled sources
        dict(_rmat(22), name="bc4_rmat22", op="bc", n=4),
    ]


def draw(rng):
    op = rng.choice(["bfs", "bfs", "dobfs", "dobfs", "grid_bfs", "sssp", "grid_sssp", "cc", "pagerank", "pagerank",
                     "bfs_multi", "sssp_multi", "bc", "bc_multi"])
    if op.startswith("grid"):
        c = _grid(int(2 ** rng.uniform(5, 11.5)), int(2 ** rng.uniform(5, 11.5)))
        if op == "grid_bfs":
            return dict(c, op="bfs", direction=rng.choice([grx.GRX_DIR_PUSH, grx.GRX_DIR_AUTO]))
        return dict(c, op="sssp", wmax=rng.choice([64, 1000]), sssp_delta=int(2 ** rng.uniform(10, 17)))
    top = {"bfs": 24, "dobfs": 24, "sssp": 23, "cc": 24, "pagerank": 24, "bfs_multi": 23, "sssp_multi": 21, "bc": 22,
           "bc_multi": 19}[op]
    scale = rng.randint(12, top)
    nv = int(2 ** rng.uniform(scale - 1, scale)) | 1
    c = _rmat(scale, rng.choice([4, 8, 16, 16]), nv)
    c["offsets64"] = op in ("bfs", "dobfs", "sssp", "pagerank") and rng.random() < 0.25
    if op == "bfs":
        return dict(c, op="bfs", direction=grx.GRX_DIR_PUSH)
    if op == "dobfs":
        return dict(c, op="bfs", alpha=10 ** rng.uniform(-5, -2), beta=10 ** rng.uniform(-2, -1),
                    exact_fv=rng.randint(0, 1))
    if op == "sssp":
        return dict(c, op="sssp", wmax=rng.choice([1, 64, 1000]))
    if op == "cc":
        return dict(c, op="cc")
    if op == "pagerank":
        return dict(c, op="pagerank", iters=rng.randint(5, 40))
    if op == "bfs_multi":
        return dict(c, op="bfs_multi", n=rng.randint(1, 64))
    if op == "sssp_multi":
        return dict(c, op="sssp_multi", wmax=64, n=rng.randint(1, 64))
    return dict(c, op=op, n=rng.randint(1, 4) if op == "bc" else rng.randint(1, 64))


def _csr(case, seed):
    """Row offsets, columns and weights (or None) of the case's graph, on the GPU."""
    if case["graph"] == "grid":
        return grx.grid_graph_device(case["width"], case["height"], 0.1, seed=seed, wmax=case.get("wmax"))
    u, v = grx.rmat_edges(case["scale"], case["ef"], seed)
    if case["nv"] < 1 << case["scale"]:
        keep = (u < case["nv"]) & (v < case["nv"])
        u, v = u[keep], v[keep]
    ro, col = grx.build_csr_device(case["nv"], u, v)
    w = grx.edge_weights(ro, col, case["wmax"], 100 + seed) if case.get("wmax") else None
    return ro, col, w


def _sources(ro, count, seed):
    """Random vertices with edges."""
    rng = random.Random(seed)
    with_edges = torch.nonzero(ro[1:] > ro[:-1]).view(-1)
    return [int(with_edges[rng.randrange(with_edges.numel())]) for _ in range(count)]


_OPTIONS = ("direction", "alpha", "beta", "exact_fv", "push_bitmap", "sssp_delta")


def prepare(case, seed):
    ro, col, w = _csr(case, seed)
    srcs = _sources(ro, case.get("n", 1), seed) if case["op"] not in ("cc", "pagerank") else None
    if not case["offsets64"]:
        ro = ro.to(torch.int32)
    g = grx.graph_load_csr(ro, col, w, offsets64=case["offsets64"])
    torch.cuda.current_stream().synchronize()      # the graph has its copies before ours go
    return {"op": case["op"], "g": g, "srcs": srcs, "iters": case.get("iters", 0),
            "opts": grx.opts(**{k: case[k] for k in _OPTIONS if k in case})}


def run(state):
    op, g, srcs, o = state["op"], state["g"], state["srcs"], state["opts"]
    if op == "bfs":
        return grx.bfs(g, srcs[0], opts=o)
    if op == "sssp":
        return grx.sssp(g, srcs[0], opts=o)
    if op == "cc":
        return grx.cc(g)
    if op == "pagerank":
        return grx.pagerank(g, 0.85, state["iters"])
    return getattr(grx, op)(g, srcs, opts=o)


def _edges(case):
    """About how many directed edges are left without loops and duplicates."""
    if case["graph"] == "grid":
        return 3.6 * case["nv"]
    s = case["scale"]
    kept = 1 - min(0.5, 0.044 * 0.825 ** (s - 22) * case["ef"] / 16)
    return 2 * case["ef"] * (1 << s) * kept * (case["nv"] / (1 << s)) ** 0.8


def work(case):
    v, e, op = case["nv"], _edges(case), case["op"]
    offsets = (8 if case["offsets64"] else 4) * (v + 1)
    if op == "bfs":       # push reads every column; a pull needs one per vertex
        cols = e if case.get("direction", grx.GRX_DIR_AUTO) == grx.GRX_DIR_PUSH or case["graph"] == "grid" else v
        return {"bytes": offsets + 4 * cols + 4 * v, "flops": 0}
    if op == "sssp":
        return {"bytes": offsets + 8 * e + 4 * v, "flops": 0}
    if op == "cc":        # two neighbours of each vertex and the labels
        return {"bytes": offsets + 8 * v + 4 * v, "flops": 0}
    if op == "pagerank":  # the columns, the old and the new ranks in every iteration
        return {"bytes": offsets + case["iters"] * (4 * e + 8 * v), "flops": case["iters"] * (e + 3 * v)}
    if op == "bfs_multi":
        return {"bytes": offsets + 4 * e + 4 * case["n"] * v, "flops": 0}
    if op == "sssp_multi":
        return {"bytes": offsets + 8 * e + 4 * case["n"] * v, "flops": 0}
    sweeps = case["n"] if op == "bc" else 1
    return {"bytes": offsets + sweeps * (4 * e + 16 * v) + 8 * v, "flops": 4 * case["n"] * e}


def _exact_pagerank(a, deg, nv, damping, iters):
    r = torch.full((nv,), 1.0 / nv, dtype=torch.float64, device=deg.device)
    lone = deg == 0
    share = torch.where(lone, torch.ones_like(deg), deg)
    for _ in range(iters):
        c = torch.where(lone, torch.zeros_like(r), r / share)
        r = (1 - damping) / nv + damping * (a @ c + r[lone].sum() / nv)
    return r


def _exact_bc(a, nv, srcs):
    bc = torch.zeros(nv, dtype=torch.float64, device=a.device)
    for s in srcs:
        sigma = torch.zeros_like(bc)
        sigma[s] = 1
        levels = [sigma != 0]
        reached = levels[0].clone()
        while True:                                   # path counts, level by level
            more = (a @ (sigma * levels[-1])) * ~reached
            found = more != 0
            if not bool(found.any()):
                break
            sigma += more
            reached |= found
            levels.append(found)
        delta = torch.zeros_like(bc)
        for k in range(len(levels) - 1, 0, -1):       # dependencies, from the deepest level back
            coef = torch.where(levels[k], (1 + delta) / torch.where(levels[k], sigma, torch.ones_like(sigma)),
                               torch.zeros_like(sigma))
            delta += (a @ coef) * sigma * levels[k - 1]
        delta[s] = 0
        bc += delta
    return bc


def exact(case, seed):
    """PageRank and betweenness in 64 bits by sparse matrix products; the other
    outputs are whole numbers."""
    if case["op"] not in ("pagerank", "bc", "bc_multi"):
        return None
    ro, col, _ = _csr(case, seed)
    a = torch.sparse_csr_tensor(ro, col.to(torch.int64), torch.ones(col.numel(), dtype=torch.float64, device=col.device),
                                size=(case["nv"], case["nv"]))
    if case["op"] == "pagerank":
        return _exact_pagerank(a, (ro[1:] - ro[:-1]).to(torch.float64), case["nv"], 0.85, case["iters"])
    return _exact_bc(a, case["nv"], _sources(ro, case["n"], seed))

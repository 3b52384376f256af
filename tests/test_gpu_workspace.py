"""Device memory of the graphs, seen through the allocator: what a refused
request leaves behind, what goes back to make room, captured calls, and how
many blocks a call ran on."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1504_04804_gb300 import build, inputs
from recording_allocator import recorded

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def grx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    oracle.build()
    from paper_1504_04804_gb300 import grx as g
    return g


# Each entry point on a graph (R-MAT or grid), and the oracle's result for it.
def _bfs(grx, dg, g, srcs):
    return grx.bfs(dg, srcs[0]).cpu().numpy(), oracle.bfs(g.row_offsets, g.col_indices, srcs[0])


def _sssp(grx, dg, g, srcs):
    return (grx.as_uint32(grx.sssp(dg, srcs[0], opts=grx.opts(sssp_delta=40))),
            oracle.sssp(g.row_offsets, g.col_indices, g.weights, srcs[0]))


def _pagerank(grx, dg, g, srcs):
    return grx.pagerank(dg, 0.85, 20).cpu().numpy(), oracle.pagerank(g.row_offsets, g.col_indices, 0.85, 20)


def _bc(grx, dg, g, srcs):
    return grx.bc(dg, srcs[:2]).cpu().numpy(), oracle.bc(g.row_offsets, g.col_indices, srcs[:2])


def _bc_multi(grx, dg, g, srcs):
    return grx.bc_multi(dg, srcs).cpu().numpy(), oracle.bc(g.row_offsets, g.col_indices, srcs)


def _bfs_multi(grx, dg, g, srcs):
    return (grx.bfs_multi(dg, srcs).cpu().numpy(),
            np.stack([oracle.bfs(g.row_offsets, g.col_indices, s) for s in srcs]))


def _sssp_multi(grx, dg, g, srcs):
    return (grx.as_uint32(grx.sssp_multi(dg, srcs)),
            np.stack([oracle.sssp(g.row_offsets, g.col_indices, g.weights, s) for s in srcs]))


def _bfs64(grx, dg, g, srcs):
    return grx.bfs64(dg, srcs[0]).cpu().numpy(), oracle.bfs(g.row_offsets, g.col_indices, srcs[0])


CALLS = {f.__name__[1:]: f for f in (_bfs, _sssp, _pagerank, _bc, _bc_multi, _bfs_multi, _sssp_multi, _bfs64)}


@pytest.fixture(scope="module")
def graphs():
    r = inputs.rmat_graph(10, 16, seed=10, wmax=64, weight_seed=11)
    t = inputs.grid_graph(61, 47, p_del=0.1, seed=4)
    t = inputs.Graph(t.name, t.row_offsets, t.col_indices, inputs.edge_weights(t.row_offsets, t.col_indices, 50, 5))
    return {"rmat": r, "grid": t}


def _load(grx, call, g):
    if call == "bfs64":
        return grx.graph_load_csr64(g.row_offsets, g.col_indices)
    return grx.load(g)


def _check(grx, call, dg, g):
    srcs = [int(s) for s in inputs.pick_sources(g.row_offsets, 5, seed=2)]
    got, want = CALLS[call](grx, dg, g, srcs)
    grx.graph_status(dg)
    if want.dtype.kind == "f":
        assert np.allclose(got, want, rtol=1e-5 if call == "pagerank" else 1e-9, atol=0)
    else:
        assert np.array_equal(got, want)


def _footprint(grx, call, dg):
    kind = {"bfs_multi": grx.GRX_KIND_BFS, "sssp_multi": grx.GRX_KIND_SSSP}.get(call)
    return None if kind is None else grx.multi_footprint(dg, kind)


@pytest.mark.parametrize("name", ["rmat", "grid"])
@pytest.mark.parametrize("call", list(CALLS))
def test_a_call_that_was_refused_memory_can_be_made_again(grx, graphs, call, name):
    """Every request of the first call refused in turn: it says GRX_ENOMEM (or does without), the second call
    gives the result, and both together hold what one call holds that was not refused."""
    g = graphs[name]
    if call == "bc_multi" and name == "grid":
        pytest.skip("deeper than bc_multi's levels")
    with recorded(grx) as mem:
        dg = _load(grx, call, g)
        first = mem.asked
        _check(grx, call, dg, g)
        requests, held = mem.asked - first, sorted(n for _, n in mem.live.values())
        dg.free()
        assert not mem.live
    assert requests > 0
    for k in range(requests):
        with recorded(grx, refuse=[first + k]) as mem:
            dg = _load(grx, call, g)
            done = True
            try:
                _check(grx, call, dg, g)
            except grx.GrxError as e:
                assert e.status == grx.GRX_ENOMEM, k
                done = False
            assert mem.refused == 1
            need, used = _footprint(grx, call, dg), mem.used()
            _check(grx, call, dg, g)
            assert need is None or mem.used() - used == need, k
            now = [n for _, n in mem.live.values()]
            for n in held:
                now.remove(n)
            assert done or not now, k                # a call that did without may keep what it used instead
            dg.free()
            assert not mem.live


FLAGS = 4096                             # entries of the grid barrier's flags: a block writes its own, block 0 none


@pytest.mark.parametrize("call,threads", [("bfs", 384), ("sssp", 384), ("bfs_multi", 384), ("sssp_multi", 256),
                                          ("bc", 384), ("bc_multi", 128), ("bfs64", 256)])
@pytest.mark.parametrize("units", [1, 2, 6, 31])
def test_grid_blocks_counts_units_of_256_threads(grx, graphs, call, threads, units):
    """As many blocks as make up grid_blocks x 256 threads, whatever the kernel's block size."""
    g = graphs["rmat"]
    with recorded(grx) as mem:
        dg = _load(grx, call, g)
        before = set(mem.live)
        srcs = [int(s) for s in inputs.pick_sources(g.row_offsets, 2, seed=2)]
        arg = srcs if call in ("bfs_multi", "sssp_multi", "bc", "bc_multi") else srcs[0]
        getattr(grx, call)(dg, arg, opts=grx.opts(grid_blocks=units))
        grx.graph_status(dg)
        (flags,) = [p for p in set(mem.live) - before if mem.live[p][1] == 4 * FLAGS]
        assert int((mem.words(flags, FLAGS) != 0).sum()) + 1 == -(-units * 256 // threads)
        dg.free()


@pytest.fixture(scope="module")
def long_grid():
    g = inputs.grid_graph(200, 203, p_del=0.1, seed=4)
    return inputs.Graph(g.name, g.row_offsets, g.col_indices,
                        inputs.edge_weights(g.row_offsets, g.col_indices, 50, 5))


def _required(grx, g):
    """Bytes that a graph, pagerank in CSR order and both multi-source calls cannot do without."""
    with recorded(grx) as mem:
        dg = grx.load(g)
        grx.pagerank(dg, 0.85, 1)
        for call in ("bfs_multi", "sssp_multi"):
            _check(grx, call, dg, g)
        used = mem.used()
        dg.free()
    return used


def test_optional_buffers_go_back_when_memory_is_refused(grx, long_grid):
    """Calls that fit a budget fit it whatever ran before them: the buffers of narrow levels, of list rounds and of
    the sorted rows make room, and those calls go on without them."""
    need = _required(grx, long_grid)
    with recorded(grx, budget=need) as mem:
        dg = grx.load(long_grid)
        grx.cc(dg)
        before = set(mem.live)
        for call in ("bfs", "sssp", "pagerank"):
            _check(grx, call, dg, long_grid)
        assert len(set(mem.live) - before) >= 3 and mem.refused == 0
        for call in ("bfs_multi", "sssp_multi"):
            _check(grx, call, dg, long_grid)
        assert mem.refused > 0
        for call in CALLS:
            if call not in ("bfs64", "bc", "bc_multi"):
                _check(grx, call, dg, long_grid)
        dg.free()
        assert not mem.live


def _captured(run):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    return graph


@pytest.mark.parametrize("warm", [False, True])
def test_calls_in_a_captured_graph(grx, long_grid, warm):
    """bfs, sssp and pagerank captured before the optional buffers are there (the capture allocates nothing and does
    without) and after (they stay, whatever is refused later); each graph is replayed for the result."""
    g = long_grid
    src = int(inputs.pick_sources(g.row_offsets, 1, seed=2)[0])
    want = {"bfs": oracle.bfs(g.row_offsets, g.col_indices, src),
            "sssp": oracle.sssp(g.row_offsets, g.col_indices, g.weights, src),
            "pagerank": oracle.pagerank(g.row_offsets, g.col_indices, 0.85, 20)}
    need = _required(grx, g)
    with recorded(grx, budget=need) as mem:
        dg = grx.load(g)
        out = {"bfs": torch.empty(g.nv, dtype=torch.int32, device="cuda"),
               "sssp": torch.empty(g.nv, dtype=torch.int32, device="cuda"),
               "pagerank": torch.empty(g.nv, dtype=torch.float32, device="cuda")}
        o = grx.opts(sssp_delta=40)
        run = {"bfs": lambda: grx.bfs(dg, src, depth_out=out["bfs"]),
               "sssp": lambda: grx.sssp(dg, src, dist_out=out["sssp"], opts=o),
               "pagerank": lambda: grx.pagerank(dg, 0.85, 20, rank_out=out["pagerank"])}
        grx.cc(dg)
        grx.pagerank(dg, 0.85, 1)
        before = set(mem.live)
        if warm:
            for f in run.values():
                f()
            assert len(set(mem.live) - before) >= 3
        live = set(mem.live)
        torch.cuda.synchronize()
        graphs = {k: _captured(f) for k, f in run.items()}
        assert set(mem.live) == live
        if warm:                                     # no room: what the graphs use is not given back
            with pytest.raises(grx.GrxError) as e:
                grx.bfs_multi(dg, [src] * 4)
                grx.sssp_multi(dg, [src] * 4)
            assert e.value.status == grx.GRX_ENOMEM and live <= set(mem.live)
        for _ in range(3):
            for k, graph in graphs.items():
                out[k].fill_(77)
                graph.replay()
                grx.graph_status(dg)
                got = out[k].cpu().numpy()
                if k == "pagerank":
                    assert np.max(np.abs(got - want[k]) / want[k]) <= 1e-5
                else:
                    assert np.array_equal(got.view(want[k].dtype), want[k]), k
        del graphs
        dg.free()


@pytest.mark.parametrize("name", ["rmat", "grid"])
@pytest.mark.parametrize("call", list(CALLS))
def test_allocators_that_align_to_eight_bytes(grx, graphs, call, name):
    """Buffers start where their types want them all the same (16-byte loads, control words on lines of 128 bytes),
    and go back by the allocator's address."""
    if call == "bc_multi" and name == "grid":
        pytest.skip("deeper than bc_multi's levels")
    with recorded(grx, skew=8) as mem:
        dg = _load(grx, call, graphs[name])
        _check(grx, call, dg, graphs[name])
        _check(grx, call, dg, graphs[name])
        dg.free()
        assert not mem.live

"""Narrow levels (a group of blocks runs the small levels of a deep graph):
traversals that go in and out of them at every limit, against the oracle,
bit-exact; parents by the oracle's checker."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1504_04804_gb300 import build, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def grx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    oracle.build()
    from paper_1504_04804_gb300 import grx as g
    return g


def _hub_path(hubs, every):
    """A path with hubs along it, each with private leaves that lead on by one more vertex."""
    n = every * (len(hubs) + 1)
    edges, nxt = [(i, i + 1) for i in range(n - 1)], n
    for k, d in enumerate(hubs):
        for _ in range(d):
            edges += [((k + 1) * every, nxt), (nxt, nxt + 1)]
            nxt += 2
    return inputs.csr_from_edges(nxt + 3, edges)


GRAPHS = {
    # rows of one piece and its edges, of the lane-written and warp-written pieces, of more pieces than a segment
    # holds (8,192 edges), of more edges than start (16,384) or stay in (32,768) narrow levels
    "hubs": lambda: _hub_path([1, 2, 3, 4, 5, 31, 32, 33, 8191, 8193, 8300, 16383, 16385, 33000], 9),
    "grid": lambda: inputs.grid_graph(301, 97, p_del=0.1, seed=5),
    "long_grid": lambda: inputs.grid_graph(3, 5001, p_del=0.05, seed=6),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("off64", [False, True])
@pytest.mark.parametrize("direction", [0, 1])
def test_bfs_through_narrow_levels(grx, name, off64, direction):
    g = GRAPHS[name]()
    dg = grx.load(g, offsets64=off64)
    for src in (0, g.nv // 2, int(inputs.pick_sources(g.row_offsets, 1, seed=3)[0])):
        want = oracle.bfs(g.row_offsets, g.col_indices, src)
        # grids smaller than the group, the limit on a wait that renews it every few levels, bitmap pushes between
        for kw in ({}, {"grid_blocks": 1}, {"grid_blocks": 3}, {"grid_blocks": 70}, {"timeout_s": 2e-4},
                   {"push_bitmap": 0.001}, {"alpha": 1e9}):
            d, p = grx.bfs(dg, src, opts=grx.opts(direction=direction, **kw), parent=True)
            if "timeout_s" in kw:
                try:
                    grx.graph_status(dg)
                except grx.GrxError as e:                     # a slow barrier may give up: then it says so
                    assert e.status == grx.GRX_ETIMEOUT
                    continue
            grx.graph_status(dg)
            d, p = d.cpu().numpy(), p.cpu().numpy()
            assert np.array_equal(d, want), (name, src, kw)
            assert oracle.check_bfs(g.row_offsets, g.col_indices, src, d, p) == 0


def _weighted(g, wmax, seed):
    w = inputs.edge_weights(g.row_offsets, g.col_indices, wmax, seed)
    return inputs.Graph(g.name, g.row_offsets, g.col_indices, w)


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("off64", [False, True])
@pytest.mark.parametrize("wmax", [1, 300])
def test_sssp_through_list_rounds(grx, name, off64, wmax):
    g = _weighted(GRAPHS[name](), wmax, 7)
    dg = grx.load(g, offsets64=off64)
    for src in (0, g.nv // 2, int(inputs.pick_sources(g.row_offsets, 1, seed=3)[0])):
        want = oracle.sssp(g.row_offsets, g.col_indices, g.weights, src)
        for delta in (0, 1, 150, 5000):
            for kw in ({}, {"grid_blocks": 1}, {"grid_blocks": 5}, {"push_bitmap": 0.001}):
                d = grx.sssp(dg, src, opts=grx.opts(sssp_delta=delta, **kw))
                grx.graph_status(dg)
                assert np.array_equal(grx.as_uint32(d), want), (name, src, delta, kw)


def test_a_new_graph_in_the_memory_of_a_freed_one(grx):
    """Words left by a freed graph's traversals are not taken for the new one's."""
    for k in range(4):
        g = _weighted(inputs.grid_graph(120 + k, 90, p_del=0.1, seed=k), 50, k)
        dg = grx.load(g)
        src = int(inputs.pick_sources(g.row_offsets, 1, seed=k)[0])
        assert np.array_equal(grx.bfs(dg, src).cpu().numpy(), oracle.bfs(g.row_offsets, g.col_indices, src))
        d = grx.sssp(dg, src, opts=grx.opts(sssp_delta=200))
        assert np.array_equal(grx.as_uint32(d), oracle.sssp(g.row_offsets, g.col_indices, g.weights, src))
        dg.free()

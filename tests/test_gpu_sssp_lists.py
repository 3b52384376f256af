"""List rounds of SSSP: rows at the edges of their pieces, rounds at the limits
of the lists, and distances that other blocks lowered in the round before,
against the oracle, bit-exact.  Each case looks into the list buffers to see
that list rounds ran at all."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1504_04804_gb300 import build, inputs
from recording_allocator import recorded

pytestmark = pytest.mark.gpu

LINES = 2 * 512 * 4                      # 32-bit words of the exchange's lines, at the head of the buffers


@pytest.fixture(scope="module")
def grx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    oracle.build()
    from paper_1504_04804_gb300 import grx as g
    return g


def _weighted(nv, edges, wmax, seed):
    g = inputs.csr_from_edges(nv, edges)
    return inputs.Graph(g.name, g.row_offsets, g.col_indices,
                        inputs.edge_weights(g.row_offsets, g.col_indices, wmax, seed))


def _rows(degrees):
    """A path through vertices of these degrees, each with leaves that lead on by one more vertex."""
    n = 5 * (len(degrees) + 1)
    edges, nxt = [(i, i + 1) for i in range(n - 1)], n
    for k, d in enumerate(degrees):
        for _ in range(d - 2):
            edges += [(5 * (k + 1), nxt), (nxt, nxt + 1)]
            nxt += 2
    return nxt + 3, edges


def _tree(widths):
    """A tree by its vertices' children per level, with every leaf of it tied to the next one by a long way round."""
    edges, level, nxt = [], [0], 1
    for w in widths:
        below = []
        for v in level:
            edges += [(v, nxt + k) for k in range(w)]
            below += range(nxt, nxt + w)
            nxt += w
        level = below
    edges += list(zip(level, level[1:]))
    return nxt, edges


GRAPHS = {
    # pieces of one to four edges, rows written by a lane (to 32 edges) and by a warp, the largest row taken
    "rows": lambda: _rows([3, 4, 5, 31, 32, 33, 63, 64]),
    # 64 rows of 64 edges found by two blocks: more pieces than a segment's 192 in a round that fits
    "full_segment": lambda: _tree([64, 63, 1, 1]),
    # rounds of 14,000, 54,000 and 130,000 edges: inside half the limit, past it, past the limit; and down again
    "limits": lambda: _tree([60, 60, 3, 4, 1]),
    "path": lambda: (4000, [(i, i + 1) for i in range(3999)]),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("off64", [False, True])
def test_list_rounds_match_oracle(grx, name, off64):
    g = _weighted(*GRAPHS[name](), wmax=40, seed=3)
    assert np.diff(g.row_offsets).max() <= 64 and g.ne < 8 * g.nv
    with recorded(grx) as mem:
        dg = grx.load(g, offsets64=off64)
        grx.cc(dg)                                   # the traversal workspace
        before = set(mem.live)
        for src in (0, g.nv // 2, g.nv - 4):
            want = oracle.sssp(g.row_offsets, g.col_indices, g.weights, src)
            for delta in (0, 30, 700):
                for kw in ({}, {"grid_blocks": 1}, {"grid_blocks": 70}, {"grid_blocks": 10000}):
                    d = grx.sssp(dg, src, opts=grx.opts(sssp_delta=delta, **kw))
                    grx.graph_status(dg)
                    assert np.array_equal(grx.as_uint32(d), want), (src, delta, kw)
        (lists,) = set(mem.live) - before
        assert int((mem.words(lists, LINES) != 0).sum()) > 0, "no list round ran"
        dg.free()


def test_a_row_past_64_edges_stays_on_the_queue(grx):
    g = _weighted(*_rows([65]), wmax=40, seed=3)
    with recorded(grx) as mem:
        dg = grx.load(g)
        grx.cc(dg)
        before = set(mem.live)
        assert np.array_equal(grx.as_uint32(grx.sssp(dg, 0)),
                              oracle.sssp(g.row_offsets, g.col_indices, g.weights, 0))
        assert set(mem.live) == before
        dg.free()


@pytest.mark.parametrize("blocks", [0, 70, 456])
def test_distances_lowered_by_other_blocks_are_seen_in_the_next_round(grx, blocks):
    """On a grid with weights of many sizes most vertices are lowered by several blocks in the round that queues
    them, and again in later rounds.  Distances read too early would leave too large ones behind."""
    g0 = inputs.grid_graph(257, 301, p_del=0.02, seed=11)
    g = inputs.Graph(g0.name, g0.row_offsets, g0.col_indices,
                     inputs.edge_weights(g0.row_offsets, g0.col_indices, 1000, 12))
    src = int(inputs.pick_sources(g.row_offsets, 1, seed=5)[0])
    want = oracle.sssp(g.row_offsets, g.col_indices, g.weights, src)
    dg = grx.load(g)
    for _ in range(20):
        d = grx.sssp(dg, src, opts=grx.opts(grid_blocks=blocks))
        grx.graph_status(dg)
        assert np.array_equal(grx.as_uint32(d), want)


FLAGS = 4096                             # entries of the grid barrier's flags: a block writes its own, block 0 none


def _uniform(nv, ne, seed):
    rng = np.random.default_rng(seed)
    return nv, rng.integers(0, nv, (ne // 2, 2)).tolist()


@pytest.mark.parametrize("nv,ne,full", [(30_000, 120_000, False), (300_000, 1_300_000, True)])
def test_large_rounds_run_on_the_whole_grid(grx, nv, ne, full):
    """A sparse graph that is not deep: ten-odd rounds of most of its edges.  The group that runs the small
    rounds on lists is 64 blocks, the others run the large ones with it."""
    g = _weighted(*_uniform(nv, ne, 7), wmax=40, seed=3)
    assert np.diff(g.row_offsets).max() <= 64 and g.ne < 8 * g.nv and (g.ne > 1 << 20) == full
    with recorded(grx) as mem:
        dg = grx.load(g)
        before = set(mem.live)
        for delta in (0, 10):
            d = grx.sssp(dg, 1, opts=grx.opts(sssp_delta=delta))
            grx.graph_status(dg)
            assert np.array_equal(grx.as_uint32(d), oracle.sssp(g.row_offsets, g.col_indices, g.weights, 1))
        new = set(mem.live) - before
        (flags,) = [p for p in new if mem.live[p][1] == 4 * FLAGS]
        blocks = int((mem.words(flags, FLAGS) != 0).sum()) + 1
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        assert blocks == 2 * sms if full else blocks == 64
        lists = [mem.words(p, LINES).view(2, 512, 4) for p in new if mem.live[p][1] > 4 * LINES
                 and mem.live[p][1] not in (4 * g.nv, 8 * g.nv)]
        assert any(x[:, :64].any() and not x[:, 64:].any() for x in lists), "no list round of 64 blocks ran"
        dg.free()


@pytest.mark.parametrize("off64", [False, True])
def test_rounds_in_equal_shares(grx, off64):
    """No hubs and many edges: rounds of a million edges and more, several tiles a warp, the last share cut short."""
    g = _weighted(*_uniform(90_000, 2_900_000, 9), wmax=40, seed=3)
    assert np.diff(g.row_offsets).max() <= 87 and g.ne >= 8 * g.nv
    dg = grx.load(g, offsets64=off64)
    want = oracle.sssp(g.row_offsets, g.col_indices, g.weights, 5)
    for delta in (0, 10):
        for kw in ({}, {"grid_blocks": 3}, {"push_bitmap": -1.0}):
            d = grx.sssp(dg, 5, opts=grx.opts(sssp_delta=delta, **kw))
            grx.graph_status(dg)
            assert np.array_equal(grx.as_uint32(d), want), (delta, kw)


def test_narrow_levels_run_where_bfs_has_many_small_ones(grx):
    """The counterpart for BFS (its results are tested with its limits elsewhere): the group's lines are used."""
    g = inputs.grid_graph(301, 97, p_del=0.1, seed=5)
    with recorded(grx) as mem:
        dg = grx.load(g)
        grx.cc(dg)
        before = set(mem.live)
        src = int(inputs.pick_sources(g.row_offsets, 1, seed=3)[0])
        assert np.array_equal(grx.bfs(dg, src).cpu().numpy(), oracle.bfs(g.row_offsets, g.col_indices, src))
        (narrow,) = set(mem.live) - before
        assert int((mem.words(narrow, 2 * 64 * 4) != 0).sum()) > 0, "no narrow level ran"
        dg.free()

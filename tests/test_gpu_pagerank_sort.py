"""PageRank's sort of the rows by degree: rows that are all alike, long rows of
one bucket beside each other, and the sizes from which chunks and the shared
table change, against 64 bits within the 1e-5 of the PageRank parity tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1504_04804_gb300 import build, inputs
from recording_allocator import recorded

pytestmark = pytest.mark.gpu

PR_TOL = 1e-5


@pytest.fixture(scope="module")
def grx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    oracle.build()
    from paper_1504_04804_gb300 import grx as g
    return g


def _ring(n, k):
    return inputs.csr_from_edges(n, [(i, (i + j) % n) for j in range(1, k + 1) for i in range(n)])


def _stars(count, leaves):
    """Stars of neighbouring centres: rows of one bucket in one warp."""
    return inputs.csr_from_edges(count * (leaves + 1), [(c, count + c * leaves + k) for c in range(count)
                                                        for k in range(leaves)])


def _mixed(n, seed):
    """Neighbouring rows of no, few and many edges."""
    rng = np.random.default_rng(seed)
    return inputs.csr_from_edges(n, [(i, int(u)) for i in range(0, n, 7)
                                     for u in rng.choice(n, int(rng.choice([1, 3, 140, 141, 150])), replace=False)
                                     if u != i])


ALIKE = {
    "ring": lambda: _ring(20_001, 3),                # one bucket, partly filled last warp
    "stars_without_units": lambda: _stars(65, 128),  # the last bucket of slice rows
    "stars_of_warp_rows": lambda: _stars(65, 129),
    "stars_of_chunks": lambda: _stars(33, 1025),
    "mixed": lambda: _mixed(3000, 5),
}


@pytest.mark.parametrize("name", list(ALIKE))
def test_rows_alike_are_sorted_once_each(grx, name):
    g = ALIKE[name]()
    dg, other = grx.load(g), grx.load(g)
    want = oracle.pagerank(g.row_offsets, g.col_indices, 0.85, 20)
    r = grx.pagerank(dg, 0.85, 20)
    assert np.max(np.abs(r.cpu().numpy().astype(np.float64) - want) / want) <= PR_TOL
    # where rows of a bucket are placed depends on timing; their sums do not
    assert torch.equal(r, grx.pagerank(other, 0.85, 20))


def _wide(grx, nv, neighbours, seed):
    """A ring, 20,000 rows of 150 edges more (four a warp) and 420 rows of 20,000 (8,400 chunks of 1,024)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def rows(ids, edges):
        u = ids.repeat_interleave(edges)
        return u, torch.randint(0, nv, (u.numel(),), device="cuda", generator=gen)

    i = torch.arange(nv, device="cuda")
    pairs = [(i, (i + k) % nv) for k in range(1, neighbours + 1)]
    pairs += [rows(torch.arange(1000, 21_000, device="cuda"), 150), rows(torch.arange(420, device="cuda") * 3, 20_000)]
    u, v = torch.cat([p[0] for p in pairs]), torch.cat([p[1] for p in pairs])
    return grx.build_csr_device(nv, u.to(torch.int32), v.to(torch.int32))


def _starred(grx, nv, hub, edges, seed):
    """A uniform random graph, vertex 3 joined to `hub` others."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    u, v = (torch.randint(0, nv, (edges,), device="cuda", generator=gen) for _ in range(2))
    k = torch.arange(hub, device="cuda") + 10
    return grx.build_csr_device(nv, torch.cat([u, torch.full_like(k, 3)]).to(torch.int32),
                                torch.cat([v, k]).to(torch.int32))


# chunks by the longest row: 600,000 edges in 587 chunks of 1,024 where others have 512
# a row with a sixteenth of a million edges and more: CSR order, whatever the iterations
@pytest.mark.parametrize("nv,hub,edges,is_sorted", [(1_000_000, 600_000, 5_000_000, True),
                                                    (700_000, 600_000, 100_000, False),
                                                    (90_000, 80_000, 100_000, True)])
def test_graphs_with_one_long_row(grx, nv, hub, edges, is_sorted):
    ro, col = _starred(grx, nv, hub, edges, 4)
    with recorded(grx) as mem:
        dg = grx.graph_load_csr(ro, col)
        grx.pagerank(dg, 0.85, 1)
        before = set(mem.live)
        r = grx.pagerank(dg, 0.85, 20)
        torch.cuda.synchronize()
        assert bool(set(mem.live) - before) == is_sorted
        want = oracle.pagerank(ro.cpu().numpy(), col.cpu().numpy(), 0.85, 20)
        assert np.max(np.abs(r.cpu().numpy().astype(np.float64) - want) / want) <= PR_TOL
        dg.free()


# 64M edges: chunks of 1,024; 2^24 rows: the smaller shared table
@pytest.mark.parametrize("nv,neighbours", [(3_000_000, 10), ((1 << 24) + 77, 2)])
def test_large_graphs_match_64_bits(grx, nv, neighbours):
    ro, col = _wide(grx, nv, neighbours, 9)
    assert col.numel() >= 64 << 20
    iters = 8
    dg, other = grx.graph_load_csr(ro, col), grx.graph_load_csr(ro, col)
    r = grx.pagerank(dg, 0.85, iters)
    a = torch.sparse_csr_tensor(ro, col.to(torch.int64), torch.ones(col.numel(), dtype=torch.float64, device="cuda"),
                                size=(nv, nv))
    deg = (ro[1:] - ro[:-1]).to(torch.float64)
    want = torch.full((nv,), 1.0 / nv, dtype=torch.float64, device="cuda")
    for _ in range(iters):
        want = 0.15 / nv + 0.85 * (a @ (want / deg))
    assert float(((r.to(torch.float64) - want).abs() / want).max()) <= PR_TOL
    assert torch.equal(r, grx.pagerank(other, 0.85, iters))

"""PageRank over degree-sorted rows: rows at the edges of its three classes
(slices of 32 rows up to 128 edges, a warp per row, chunks), against the FP64
oracle within the 1e-5 of the PageRank parity tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1504_04804_gb300 import build, inputs

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


def _hubs(degrees, spare):
    """Hubs with private leaves, and `spare` isolated vertices at the end."""
    edges, leaf = [], len(degrees)
    for h, d in enumerate(degrees):
        edges += [(h, leaf + k) for k in range(d)]
        leaf += d
    return inputs.csr_from_edges(leaf + spare, edges)


SIZES = {
    # unit, slice, warp-row, chunk (128 edges on a graph this small) and long-row (1,024) edges
    "class_edges": lambda: _hubs([1, 2, 3, 4, 5, 127, 128, 129, 130, 255, 256, 257, 1023, 1024, 1025, 1151, 1152, 1153,
                                  5000, 9001], 3),
    "one_edge": lambda: inputs.csr_from_edges(2, [(0, 1)]),
    "one_slice": lambda: _hubs([5] * 5, 0),          # 30 rows, 5 of them wider
    "one_slice_and_a_row": lambda: _hubs([31, 1], 1),
    "rmat18": lambda: inputs.rmat_graph(18, 16, seed=18),    # chunks of 256 edges, c past the shared table
}


@pytest.mark.parametrize("name", list(SIZES))
@pytest.mark.parametrize("off64", [False, True])
def test_sorted_rows_match_oracle(grx, name, off64):
    g = SIZES[name]()
    dg = grx.load(g, offsets64=off64)
    # 3: CSR order (too few iterations to sort for); 20: sorts; 2: sorted already
    for iters in (3, 20, 2):
        r = grx.pagerank(dg, 0.85, iters).cpu().numpy().astype(np.float64)
        want = oracle.pagerank(g.row_offsets, g.col_indices, 0.85, iters)
        assert np.max(np.abs(r - want) / want) <= PR_TOL, (name, iters)
    again = grx.pagerank(dg, 0.85, 20)
    assert torch.equal(again, grx.pagerank(dg, 0.85, 20))    # sums do not depend on timing

"""Multi-source BFS, pull levels: rows on both sides of what a lane (2 edges),
eight lanes (128), a warp (2,048) and a piece (1,024 after 128) take, and, on
graphs of few edges a vertex, a lane (10); a few rows and 128 at a time, against
the oracle, bit-exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1504_04804_gb300 import build, inputs

pytestmark = pytest.mark.gpu

DEGREES = [1, 2, 3, 5, 6, 7, 9, 10, 11, 12, 33, 34, 35, 66, 127, 128, 129, 130, 383, 384, 385, 1151, 1152, 1153, 2047, 2048, 2049, 2175, 2176,
           2177, 3200]


@pytest.fixture(scope="module")
def grx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    oracle.build()
    from paper_1504_04804_gb300 import grx as g
    return g


def _hubs(spare, dense):
    """Hubs of DEGREES among leaves of their own; leaves number i of neighbouring hubs are joined now and then, so
    that lanes reach a hub through its first, middle and last neighbours, some levels apart."""
    edges, first, nxt = [], [], len(DEGREES)
    for h, d in enumerate(DEGREES):
        first.append(nxt)
        edges += [(h, nxt + k) for k in range(d)]
        nxt += d
    for h in range(len(DEGREES) - 1):
        a, b = DEGREES[h], DEGREES[h + 1]
        edges += [(first[h] + a - 1, first[h + 1] + b - 1), (first[h] + a // 2, first[h + 1])]
    ends = [first[h] + k for h, d in enumerate(DEGREES) for k in (0, d // 2, d - 1)]
    if dense:                                    # more than eight edges a vertex on the whole
        edges += [(nxt + i, nxt + j) for i in range(450) for j in range(i)]
        ends += [nxt, nxt + 449]
        nxt += 450
    return inputs.csr_from_edges(nxt + spare, edges), ends


@pytest.mark.parametrize("spare", [0, 1])            # outputs whose lanes start on 16-byte boundaries, or not
@pytest.mark.parametrize("dense", [False, True])
@pytest.mark.parametrize("off64", [False, True])
def test_pull_rows_match_oracle(grx, off64, dense, spare):
    g, ends = _hubs(0, dense)
    g, ends = _hubs(-g.nv % 4 + spare, dense)
    assert (g.ne >= 8 * g.nv) == dense
    srcs = (ends + list(range(len(DEGREES))))[-64:]
    want = np.stack([oracle.bfs(g.row_offsets, g.col_indices, s) for s in srcs])
    dg = grx.load(g, offsets64=off64)
    for n in (1, 31, 33, 64):
        for kw in ({"direction": 2}, {"direction": 2, "grid_blocks": 1}, {"alpha": 1e-9, "beta": 1e-9}, {}):
            got = grx.bfs_multi(dg, srcs[:n], opts=grx.opts(**kw))
            grx.graph_status(dg)
            assert np.array_equal(got.cpu().numpy(), want[:n]), (n, kw)

"""Connected components by the form the graph's size and largest degree choose
(blocks of 256 or 1,024 threads, one or two vertices in flight), against the
oracle, bit-exact; the grid barrier's flags tell the block size."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1504_04804_gb300 import build, inputs
from recording_allocator import recorded

pytestmark = pytest.mark.gpu

FLAGS = 4096                             # entries of the grid barrier's flags: a block writes its own, block 0 none
LINE = 1 << 17                           # vertices from which graphs without hubs take the smaller blocks


@pytest.fixture(scope="module")
def grx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    oracle.build()
    from paper_1504_04804_gb300 import grx as g
    return g


def _ring(n, k, cut=7):
    """n vertices on a ring with k neighbours each side, cut into `cut` arcs, the last vertex alone."""
    i = np.arange(n - 1)
    e = [np.stack([i[:-j], i[j:]], 1)[(i[:-j] * cut // n) == (i[j:] * cut // n)] for j in range(1, k + 1)]
    return inputs.csr_from_edges(n, np.concatenate(e).tolist())


def _hub(n, d):
    """A path of n vertices, vertex 5 joined to d others."""
    edges = [(i, i + 1) for i in range(n - 2)] + [(5, 10 + 2 * k) for k in range(d - 2)]
    return inputs.csr_from_edges(n, edges)


CASES = {
    "path_at_the_line": (lambda: _ring(LINE, 1), 1024),
    "path_past_the_line": (lambda: _ring(LINE + 1, 1), 256),
    "dense_ring": (lambda: _ring(150_001, 6), 256),
    "hub_of_a_thousandth": (lambda: _hub(LINE + 1, 128), 256),
    "hub_of_more": (lambda: _hub(LINE + 1, 129), 1024),
    "rmat": (lambda: inputs.rmat_graph(17, 8, seed=3), 1024),
    "rmat_dense": (lambda: inputs.rmat_graph(14, 16, seed=3), 1024),
}


@pytest.mark.parametrize("name", list(CASES))
def test_labels_and_blocks(grx, name):
    make, threads = CASES[name]
    g = make()
    with recorded(grx) as mem:
        dg = grx.load(g)
        before = set(mem.live)
        assert np.array_equal(grx.cc(dg).cpu().numpy(), oracle.cc(g.row_offsets, g.col_indices))
        grx.graph_status(dg)
        # (bitmaps of as many bytes come before the flags)
        flags = [p for p in mem.live if p not in before and mem.live[p][1] == 4 * FLAGS][-1]
        blocks = int((mem.words(flags, FLAGS) != 0).sum()) + 1
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        assert (blocks > 2 * sms) == (threads == 256), blocks
        dg.free()

"""The passes over the arcs at the edges of their pieces (steps of 128 arcs, 32
row ends a turn): arc counts around multiples of a step, long rows, and runs of
more than 32 vertices without arcs before, between and after them. The labels
equal the oracle's, and a fault in the first or last arc is still found.
Integers: comparisons are exact."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1907_00140_gb300 as chl  # noqa: E402
from test_gpu_parity import DG, assert_same, dev, gpu_labels  # noqa: E402
from test_gpu_query_blocks import graph_of  # noqa: E402


def stars(leaves, gap, seed):
    """Two stars of the given sizes; `gap` isolated vertices before, between and
    after every centre's leaves."""
    rng = np.random.default_rng(seed)
    a, b, at = [], [], gap
    for k in leaves:
        a.append(np.full(k, at))
        b.append(at + 1 + gap + np.arange(k))
        at += 1 + gap + k + gap
    a, b = np.concatenate(a), np.concatenate(b)
    g = graph_of(at, a, b, rng.integers(1, 100, len(a)))
    return g, rng.permutation(at).astype(np.uint32)


@pytest.mark.parametrize("leaves", [(1,), (16, 15), (32, 32), (63,), (64,), (65,), (127, 1), (500, 524), (3000, 70)])
@pytest.mark.parametrize("gap", [0, 31, 32, 33, 100])
def test_arc_counts_and_empty_rows(leaves, gap):
    g, rank = stars(leaves, gap, seed=sum(leaves) + gap)
    assert len(g.col) == 2 * sum(leaves)
    assert_same(O.build_labels(g, rank, "pll"), *gpu_labels(g, rank)[1:4])


@pytest.mark.parametrize("at", [0, -1])
@pytest.mark.parametrize("fault", ["weight", "id", "order", "reverse"])
def test_faults_at_the_ends(at, fault):
    g, rank = stars((127, 65), 33, seed=7)
    d = DG(g)
    if fault == "weight":
        d.w[at] = 0
    elif fault == "id":
        d.col[at] = g.n
    elif fault == "reverse":
        d.w[at] += 1
    else:  # the first and the last row of several arcs, back to front
        v = np.flatnonzero(np.diff(g.row_ptr.astype(np.int64)) > 1)[at]
        x, y = int(g.row_ptr[v]), int(g.row_ptr[v + 1])
        d.col[x:y] = d.col[x:y].flip(0)
        d.w[x:y] = d.w[x:y].flip(0)
    with pytest.raises(chl.ChlError, match="invalid graph"):
        chl.build_labels(d, dev(rank))

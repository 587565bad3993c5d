"""The passes over the arcs at the edges of their pieces (steps of 128 arcs, 32
row ends a turn): arc counts around multiples of a step, long rows, and runs of
more than 32 vertices without arcs before, between and after them. The labels
equal the oracle's, and a fault in the first or last arc is still found.
Integers: comparisons are exact."""
import numpy as np
import pytest

import oracle as O
import workloads as W

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


def test_long_run_of_empty_rows():
    """Ten million isolated vertices between the arcs, in the caller's numbering and
    in rank order: the checks and the renumbering take about as long as with the
    isolated vertices at the end of both, and the labels are the same ones."""
    m, gap = 2000, 10_000_000
    n, rng = m + gap, np.random.default_rng(11)
    i = np.arange(m - 1)
    i = i[i % 7 != 3]
    w = rng.integers(1, 100, len(i))
    order = rng.permutation(m)
    prep, labels = {}, {}
    for at in (m, m // 2):  # the isolated vertices follow vertex and position `at`
        def moved(v):
            return np.where(v < at, v, v + gap)

        pos = np.empty(n, np.int64)
        core = moved(np.arange(m))
        rest = np.arange(at, at + gap)
        pos[core] = moved(order)
        pos[rest] = rest
        rank = (n - 1 - pos).astype(np.uint32)
        s, t = moved(np.concatenate([i, i + 1])), moved(np.concatenate([i + 1, i]))
        o = np.lexsort((t, s))
        row = np.zeros(n + 1, np.uint64)
        row[1:] = np.cumsum(np.bincount(s, minlength=n))
        g = W.Graph(n, row, t[o].astype(np.uint32), np.concatenate([w, w])[o].astype(np.uint32))
        d, r = DG(g), dev(rank)
        for _ in range(2):
            L = chl.build_labels(d, r, slots=8, label_capacity=12_000_000)
            st = L.stats()
            prep[at] = st["build_ms"] - st["tree_ms"] - st["sort_ms"]
            off, hub, dist = L.to_numpy()
            L.free()
        first = off[core].astype(np.int64)
        length = off[core + 1].astype(np.int64) - first
        take = np.repeat(first - np.cumsum(length) + length, length) + np.arange(length.sum())
        back = np.where(hub[take] < at, hub[take], hub[take].astype(np.int64) - gap)
        labels[at] = (length, back, dist[take])
        assert len(hub) == length.sum() + gap
    for x, y in zip(*labels.values()):
        assert np.array_equal(x, y)
    assert prep[m // 2] < 3 * prep[m] + 10, prep  # (0.9 ms at the end; 188 in the middle when a warp walked them)

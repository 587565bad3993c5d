"""The query kernels at the edges of their blocks: label lists of one entry
less, as many and one more than a chunk (32) and a block (128) hold, hub
positions that share a slot of the 1,024-slot lookup table, and paths whose
walked side is longer than the buffer that keeps it (512 vertices), against
the oracle. Integers: comparisons are exact."""
import numpy as np
import pytest

import oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1907_00140_gb300 as chl  # noqa: E402
from test_gpu_parity import DG, dev  # noqa: E402


def graph_of(n, a, b, w):
    """Symmetric CSR of the undirected edges (a[i], b[i]) of weight w[i]."""
    s, t, ww = np.concatenate([a, b]), np.concatenate([b, a]), np.concatenate([w, w])
    o = np.lexsort((t, s))
    row = np.concatenate([[0], np.cumsum(np.bincount(s, minlength=n))]).astype(np.uint64)
    return W.Graph(n, row, t[o].astype(np.uint32), ww[o].astype(np.uint32))


def two_centres(m, stride, seed):
    """Two lowest-ranked centres joined to the same m leaves: both centres'
    lists hold every leaf (a detour is longer than any edge). Leaf i has rank
    position i * stride; pendant vertices at the top leaf take the positions
    between, so that the leaves of a list lie `stride` positions apart."""
    rng = np.random.default_rng(seed)
    fill = m * stride - m
    n = 2 + m + fill
    leaf = np.arange(2, 2 + m)
    filler = np.arange(2 + m, n)
    a = np.concatenate([np.zeros(m), np.ones(m), np.full(fill, 2)]).astype(np.int64)
    b = np.concatenate([leaf, leaf, filler])
    w = rng.integers(1000, 2000, len(a))
    pos = np.empty(n, np.int64)
    pos[leaf] = np.arange(m) * stride
    free = np.setdiff1d(np.arange(m * stride), pos[leaf])
    pos[filler] = free
    pos[0], pos[1] = n - 2, n - 1
    return graph_of(n, a, b, w), (n - 1 - pos).astype(np.uint32), leaf


@pytest.mark.parametrize("m,stride", [(1, 1), (31, 1), (32, 1), (127, 1), (128, 1), (129, 1), (300, 1),
                                      (130, 512), (140, 1024), (70, 300)])
def test_list_lengths_and_shared_slots(m, stride):
    g, rank, leaf = two_centres(m, stride, seed=m)
    ref = O.build_labels(g, rank, "plant", threads=8)
    assert int(ref.offsets[1] - ref.offsets[0]) >= m + 1
    L = chl.build_labels(DG(g), dev(rank))
    some = np.concatenate([[0, 1], leaf[:40], leaf[-40:], np.arange(max(2, g.n - 20), g.n)])
    pairs = np.array([(u, v) for u in some for v in some], np.uint32)
    want = O.query(ref, rank, pairs)
    assert np.array_equal(L.query(dev(pairs)).cpu().numpy().view(np.uint32), want)
    assert np.array_equal(L.query(pairs, grouped=True), want)
    cuts = sorted({0, max(1, m // 2), max(1, (m * stride) // 2), g.n})
    parts = [chl.build_labels(DG(g), dev(rank), root_begin=x, root_end=y) for x, y in zip(cuts, cuts[1:])]
    assert np.array_equal(chl.query_partitioned(parts, pairs), want)


def test_long_side_of_a_path():
    """A line ranked from one end: the hub of (0, v) is 0, so the v side is the
    whole path; both orders and lengths around the 512 vertices kept."""
    n = 640
    a = np.arange(n - 1)
    g = graph_of(n, a, a + 1, np.random.default_rng(3).integers(1, 50, n - 1))
    rank = np.arange(n - 1, -1, -1).astype(np.uint32)
    L = chl.build_labels(DG(g), dev(rank), flags=chl.CHL_FLAG_PARENTS)
    ends = [1, 2, 511, 512, 513, 514, 639]
    pairs = np.array([(0, v) for v in ends] + [(v, 0) for v in ends] + [(600, v) for v in ends] + [(5, 5)], np.uint32)
    for max_len in (n, 100):
        got, lens = L.paths(pairs, max_len=max_len)
        for i, (u, v) in enumerate(pairs.tolist()):
            want = list(range(u, v + 1)) if u <= v else list(range(u, v - 1, -1))
            assert int(lens[i]) == len(want)
            assert got[i, :min(len(want), max_len)].tolist() == want[:max_len]


@pytest.mark.parametrize("mode", ["merge", "grouped", "parts"])
@pytest.mark.parametrize("pinned", [True, False])
def test_host_pairs_are_read_in_stream_order(mode, pinned):
    """Pairs in pinned memory that an earlier copy on the call's stream fills: the
    call answers what the copy brings; pageable pairs give the same while the
    stream is busy."""
    g, rank, leaf = two_centres(40, 1, seed=4)
    ref = O.build_labels(g, rank, "plant", threads=8)
    pairs = np.random.default_rng(5).integers(0, g.n, (64, 2)).astype(np.uint32)
    want = O.query(ref, rank, pairs)
    assert (want != 0).any()
    L = chl.build_labels(DG(g), dev(rank))
    cut = [chl.build_labels(DG(g), dev(rank), root_begin=a, root_end=b) for a, b in ((0, 20), (20, g.n))]
    src, big = dev(pairs), torch.randn(4096, 4096, device="cuda")
    work = torch.cuda.Stream()
    host = torch.zeros(64, 2, dtype=torch.int32, pin_memory=True)
    torch.cuda.synchronize()
    with torch.cuda.stream(work):
        for _ in range(20):
            big @ big
        host.copy_(src, non_blocking=True)
    p = host.numpy().view(np.uint32) if pinned else pairs
    got = (chl.query_partitioned(cut, p, stream=work.cuda_stream) if mode == "parts"
           else L.query(p, stream=work.cuda_stream, grouped=mode == "grouped"))
    assert np.array_equal(got, want)

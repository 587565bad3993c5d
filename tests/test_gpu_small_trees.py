"""Trees built in shared memory (phases of many tiny trees) and rows relaxed by
one thread (graphs of degree at most 8), against the oracle: every key layout,
trees that outgrow the table (spilled to the general kernel, and counted once),
roots with more table labels than their hash holds, and a label buffer that
fills up while spilled roots wait. Integers: comparisons are exact."""
import re

import numpy as np
import pytest

import oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1907_00140_gb300 as chl  # noqa: E402
from test_gpu_parity import DG, dev, assert_same  # noqa: E402
from test_gpu_query_blocks import graph_of  # noqa: E402


def line_and_triples(line, triples, seed):
    """A path ranked from one end to the other, its vertices spread over all
    rank positions (the tree of its j-th vertex reaches the line - j after it,
    whose lists hold all j before it), and many paths of three vertices."""
    rng = np.random.default_rng(seed)
    n = line + 3 * triples
    a = np.concatenate([np.arange(line - 1), line + np.arange(triples) * 3, line + np.arange(triples) * 3 + 1])
    b = a + 1
    pos = np.empty(n, np.int64)
    at = np.linspace(0, n - 1, line).astype(np.int64)
    pos[:line] = at
    pos[line:] = rng.permutation(np.setdiff1d(np.arange(n), at))
    return graph_of(n, a, b, rng.integers(1, 60, len(a))), (n - 1 - pos).astype(np.uint32)


def case(name):
    if name == "line":
        return line_and_triples(1500, 22000, seed=4)  # keeps its numbering, prunes by labels
    if name == "ba40k":
        g = W.barabasi_albert(40000, 2, seed=9, wlo=1, whi=100)
        return g, W.degree_rank(g)
    if name == "rmat16":
        g = W.rmat(16, 4, seed=16, wlo=1, whi=255)
        return g, W.degree_rank(g)
    g = W.grid(280, 15600, seed=24)
    return g, W.spt_count_rank(g, 16, seed=24)


@pytest.fixture(scope="module", params=["line", "ba40k", "rmat16", "grid280"])
def built(request):
    g, rank = case(request.param)
    return request.param, g, rank, O.build_labels(g, rank, "plant", threads=8)


@pytest.mark.parametrize("opts", [dict(), dict(flags=chl.CHL_FLAG_WIDE_KEYS), dict(flags=chl.CHL_FLAG_PARENTS),
                                  dict(label_capacity=50000), dict(slots=40)],
                         ids=["default", "wide", "parents", "full buffer", "slots"])
def test_small_trees_equal_oracle(built, opts, capfd, monkeypatch):
    name, g, rank, ref = built
    monkeypatch.setenv("CHL_TRACE", "1")
    capfd.readouterr()
    L = chl.build_labels(DG(g), dev(rank), **opts)
    seen = [(int(c), int(s)) for c, s in re.findall(r"class (-?\d+) spilled (\d+)", capfd.readouterr().err)]
    assert_same(ref, *L.to_numpy())
    assert any(c >= 0 for c, _ in seen), seen  # the shared-memory kernel ran (its class depends on tree sizes)
    if name == "line" and "label_capacity" not in opts:  # (a phase built again reports its last attempt)
        assert any(s > 100 for _, s in seen), seen
    if opts.get("flags") == chl.CHL_FLAG_PARENTS and name == "line":
        off, hub, _ = L.to_numpy()
        par = L.parents()
        for v in (1, 700, 1499):  # the parent on a line ranked from its start is the vertex before
            a, b = int(off[v]), int(off[v + 1])
            assert np.array_equal(par[a:b], np.where(hub[a:b] == v, v, v - 1))


def test_full_buffer_while_spilled_roots_wait(capfd, monkeypatch):
    """The label buffer fills up in the shared-memory launch of a phase: the roots
    spilled by then are claimed by no launch and built after the buffer has grown."""
    g, rank = case("line")
    ref = O.build_labels(g, rank, "plant", threads=8)
    monkeypatch.setenv("CHL_TRACE", "1")
    capfd.readouterr()
    chl.build_labels(DG(g), dev(rank)).free()
    phases = [[int(x) for x in m] for m in re.findall(
        r"roots \[(\d+), (\d+)\).* class (-?\d+) spilled (\d+) .* labels (\d+) rounds", capfd.readouterr().err)]
    k = max((i for i, p in enumerate(phases) if p[2] >= 0), key=lambda i: phases[i][3])
    assert phases[k][3] > 100, phases
    # room for the phase's trivial roots and for few of the others
    room = sum(p[4] for p in phases[:k]) + phases[k][1] - phases[k][0]
    L = chl.build_labels(DG(g), dev(rank), label_capacity=room)
    waited = [int(x) for x in re.findall(r"(\d+) spilled ones wait", capfd.readouterr().err)]
    assert any(waited), (waited, phases)
    assert_same(ref, *L.to_numpy())


def test_spilled_trees_are_counted_once(capfd, monkeypatch):
    """On paths every vertex of a tree is expanded once, so without label pruning
    (and with one table throughout) the statistics do not depend on the kernel."""
    g, rank = case("line")
    monkeypatch.setenv("CHL_TRACE", "1")
    fixed = dict(switch_ratio=-1.0, psi_threshold=1e9, common_hubs=16)
    got = []
    for opts in (fixed, dict(fixed, small_threads_per_tree=256)):
        capfd.readouterr()
        st = chl.build_labels(DG(g), dev(rank), **opts).stats()
        seen = [(int(c), int(s)) for c, s in re.findall(r"class (-?\d+) spilled (\d+)", capfd.readouterr().err)]
        got.append(({k: st[k] for k in ("trees", "trivial", "labels", "expanded", "arcs", "pruned")}, seen))
    assert any(c >= 0 and s > 100 for c, s in got[0][1]) and all(c < 0 for c, _ in got[1][1]), got
    assert got[0][0] == got[1][0]


@pytest.mark.parametrize("tpt", [32, 64, 128, 256, 512, 1024])
@pytest.mark.parametrize("flags", [0, chl.CHL_FLAG_WIDE_KEYS, chl.CHL_FLAG_PARENTS])
def test_short_rows_every_block_size(tpt, flags):
    """Degrees 1 to 8 and a row length of 8 exactly: every block size and key layout."""
    rng = np.random.default_rng(5)
    n, deg = 3000, np.zeros(3000, np.int64)
    e = set()
    for u, v in rng.integers(0, n, (20000, 2)).tolist():
        if u != v and deg[u] < 8 and deg[v] < 8 and (min(u, v), max(u, v)) not in e:
            e.add((min(u, v), max(u, v)))
            deg[u] += 1
            deg[v] += 1
    a, b = np.array(sorted(e)).T
    g = graph_of(n, a, b, rng.integers(1, 30, len(a)))
    assert deg.max() == 8 and deg.min() < 8
    rank = W.degree_rank(g)
    ref = O.build_labels(g, rank, "plant", threads=8)
    L = chl.build_labels(DG(g), dev(rank), threads_per_tree=tpt, flags=flags)
    assert_same(ref, *L.to_numpy())


def short_rows(name):
    rng = np.random.default_rng(17)
    if name == "tree":  # wide trees: a complete binary tree in heap order, ranked by depth
        n = 2**18 - 1
        i = np.arange(1, n)
        return graph_of(n, (i - 1) // 2, i, rng.integers(1, 50, n - 1)), np.arange(n - 1, -1, -1).astype(np.uint32)
    g = W.grid(100 if name == "small mixed grid" else 150, 100, seed=5)
    u, v, w = (x.astype(np.int64) for x in g.edges())
    if name == "heavy grid":
        w = np.exp(rng.random(len(w)) * np.log(100_000)).astype(np.int64) + 1
    new = np.arange(g.n) if name in ("grid", "heavy grid") else rng.permutation(g.n)
    rank = np.empty(g.n, np.uint32)
    rank[new] = W.spt_count_rank(g, 16, seed=5)
    return graph_of(g.n, new[u], new[v], w), rank


# threads per tree in the first phase, in the later ones, in a build of a root range with and without a table
@pytest.mark.parametrize("name,first,later,ranged,bare", [
    ("grid", 128, 128, 128, 128), ("small mixed grid", 128, 128, 128, 128), ("mixed grid", 1024, 128, 128, 1024),
    ("tree", 1024, 1024, 1024, 1024), ("heavy grid", 512, 512, 512, 512)])
def test_block_size_of_short_rows(name, first, later, ranged, bare, capfd, monkeypatch):
    """Local numberings and small graphs take few threads per tree, other graphs
    once their first trees have shown that they are narrow, heavy-tailed weights the
    general rule."""
    g, rank = short_rows(name)
    ref = O.build_labels(g, rank, "plant", threads=8)
    d, r = DG(g), dev(rank)
    monkeypatch.setenv("CHL_TRACE", "1")

    def threads(**opts):
        capfd.readouterr()
        L = chl.build_labels(d, r, small_tree_expansions=1, **opts)
        return L, [int(x) for x in re.findall(r" threads (\d+) ", capfd.readouterr().err)]

    L, seen = threads()
    assert len(seen) > 1 and seen[0] == first and set(seen[1:]) == {later}, seen
    assert_same(ref, *L.to_numpy())
    for opts, want in ((dict(), ranged), (dict(common_hubs=-1), bare)):
        L, seen = threads(root_begin=100, root_end=2000, **opts)
        assert seen == [want], (seen, opts)
        off, hub, dist = L.to_numpy()
        pos = g.n - 1 - rank.astype(np.int64)
        v = np.repeat(np.arange(g.n), np.diff(ref.offsets.astype(np.int64)))
        on = (pos[ref.hub] >= 100) & (pos[ref.hub] < 2000)
        assert np.array_equal(hub, ref.hub[on]) and np.array_equal(dist, ref.dist[on])
        assert np.array_equal(np.diff(off.astype(np.int64)), np.bincount(v[on], minlength=g.n))


@pytest.mark.parametrize("per_sm,want", [(0.1, 1024), (1, 1024), (1.5, 512), (2, 512), (3, 256), (4, 256), (5, 128)])
def test_block_size_at_a_limit_of_trees(per_sm, want, capfd, monkeypatch):
    """A grid large enough to keep its numbering: few trees in flight take more threads each."""
    g, rank = case("grid280")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    monkeypatch.setenv("CHL_TRACE", "1")
    capfd.readouterr()
    L = chl.build_labels(DG(g), dev(rank), slots=int(per_sm * sms), root_end=3000, small_tree_expansions=1)
    assert set(re.findall(r" threads (\d+) ", capfd.readouterr().err)) == {str(want)}
    whole = chl.build_labels(DG(g), dev(rank), root_end=3000)
    for x, y in zip(whole.to_numpy(), L.to_numpy()):
        assert np.array_equal(x, y)


def test_label_buffer_of_large_road_like_graphs(capfd, monkeypatch):
    """Four grids of 420 x 420 side by side (about 390 labels per vertex): the label
    buffer holds them at once, so that no tree is built twice; the labels are those
    of one grid."""
    g = W.grid(420, 35_000, seed=42)
    u, v, w = (x.astype(np.int64) for x in g.edges())
    rank = W.spt_count_rank(g, 16, seed=42).astype(np.int64)
    one = chl.build_labels(DG(g), dev(rank.astype(np.uint32)))
    k = np.repeat(np.arange(4), len(u)) * g.n
    four = graph_of(4 * g.n, np.tile(u, 4) + k, np.tile(v, 4) + k, np.tile(w, 4))
    assert four.n * 512 * 12 > 4 << 30
    rank4 = (4 * np.tile(rank, 4) + np.repeat(np.arange(4), g.n)).astype(np.uint32)
    monkeypatch.setenv("CHL_TRACE", "1")
    capfd.readouterr()
    L = chl.build_labels(DG(four), dev(rank4))
    assert "label buffer full" not in capfd.readouterr().err
    st = L.stats()
    assert st["trees"] == four.n and st["labels"] == 4 * one.total > 256 * four.n
    off, hub, dist = one.to_numpy()
    off4, hub4, dist4 = L.to_numpy()
    for i in (0, 3):
        a, b = int(off4[i * g.n]), int(off4[(i + 1) * g.n])
        assert np.array_equal(hub4[a:b] - np.uint32(i * g.n), hub) and np.array_equal(dist4[a:b], dist)


@pytest.mark.parametrize("fixed,numbering", [(dict(), "the caller's numbering"),
                                             (dict(threads_per_tree=512), "rank order")])
def test_tuning_trials_run_the_kernels_of_the_build(fixed, numbering, capfd, monkeypatch):
    """A graph that a build keeps in the caller's numbering is tuned in it."""
    g, rank = case("grid280")
    d, r = DG(g), dev(rank)
    monkeypatch.setenv("CHL_TRACE", "1")
    capfd.readouterr()
    opts, rep = chl.tune(d, r, **fixed)
    assert re.findall(r"chl tune trials in (.*)", capfd.readouterr().err) == [numbering]
    want, got = chl.build_labels(d, r), chl.build_labels(d, r, **opts)
    for x, y in zip(want.to_numpy(), got.to_numpy()):
        assert np.array_equal(x, y)

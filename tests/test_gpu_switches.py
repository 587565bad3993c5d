"""GPU parity across the hybrid's switch points (Sec. 5.2): wherever the
first-phase switch (labels per arc, switch_ratio), the Psi switch
(psi_threshold), the small-tree switch (small_tree_expansions) and the
narrow bucket width after big trees (big_tree_bucket_delta) fire, and with or
without the next phase's first trees overlapped with a phase's tail
(overlap_phases), the labels are the canonical ones, bit-exact with the CPU
oracle. Only the amount
of work changes: the label table of earlier phases covers a rank-closed hub
set whenever it is used (Sec. 5.3), and the small-tree launch runs the same
search in smaller blocks. Each build's statistics show which switch fired.
"""
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

NEVER_SMALL = 1               # no tree averages fewer than one expansion
ALWAYS_SMALL = 0xFFFFFFFF     # every label-pruned phase's trees average fewer


@pytest.fixture(scope="module", autouse=True)
def _built():
    chl.build()
    chl.lib()


def _family(name):
    if name == "ba2k":
        g, rank = W.load("ba2k")
    else:
        g = W.rmat(13, 16, seed=13, whi=255)
        rank = W.degree_rank(g)
    return g, rank, O.build_labels(g, rank, "plant", threads=8)


@pytest.fixture(scope="module", params=["ba2k", "rmat13"])
def family(request):
    g, rank, ref = _family(request.param)
    return request.param, g, rank, ref, DG(g), dev(rank)


# (options, check of the build's statistics)
SWEEP = [
    # first-phase switch on labels per arc: off, never reached, default, always
    (dict(switch_ratio=-1.0), None),
    (dict(switch_ratio=1e-6, psi_threshold=1e9), lambda s: s["label_table_phases"] == 0),
    (dict(), None),
    (dict(switch_ratio=1e6), lambda s: s["label_table_phases"] == s["phases"] - 1),
    # the Psi switch alone (first-phase switch off)
    (dict(switch_ratio=-1.0, psi_threshold=0.5), lambda s: s["label_table_phases"] == s["phases"] - 1),
    (dict(switch_ratio=-1.0, psi_threshold=2.0), None),
    (dict(switch_ratio=-1.0, psi_threshold=1e9), lambda s: s["label_table_phases"] == 0),
    # the small-tree switch: never, default, right after the first label-pruned phase
    (dict(switch_ratio=1e6, small_tree_expansions=NEVER_SMALL), lambda s: s["small_tree_phases"] == 0),
    (dict(switch_ratio=1e6, small_tree_expansions=2048), None),
    (dict(switch_ratio=1e6, small_tree_expansions=ALWAYS_SMALL),
     lambda s: s["small_tree_phases"] == s["label_table_phases"] - 1),
    (dict(switch_ratio=1e6, small_tree_expansions=ALWAYS_SMALL, small_threads_per_tree=64),
     lambda s: s["small_tree_phases"] == s["label_table_phases"] - 1),
    (dict(switch_ratio=1e6, small_tree_expansions=ALWAYS_SMALL, small_threads_per_tree=1024,
          pruned_threads_per_tree=256), lambda s: s["small_tree_phases"] == s["label_table_phases"] - 1),
    # the narrow bucket width after big trees: default, off, set
    (dict(switch_ratio=1e6, big_tree_bucket_delta=-1), None),
    (dict(switch_ratio=1e6, big_tree_bucket_delta=1), None),
    (dict(switch_ratio=1e6, big_tree_bucket_delta=3, pruned_bucket_delta=4096), None),
    # the next phase's first trees in a phase's tail (second stream, older
    # table): off; in every label-pruned phase; with a label buffer so small
    # that their trees overflow it and are built again by their own phase
    (dict(switch_ratio=1e6, overlap_phases=-1), None),
    (dict(switch_ratio=1e6, small_tree_expansions=NEVER_SMALL), lambda s: s["small_tree_phases"] == 0),
    (dict(switch_ratio=1e6, small_tree_expansions=NEVER_SMALL, label_capacity=1000), None),
    (dict(switch_ratio=1e6, small_tree_expansions=NEVER_SMALL, threads_per_tree=256, flags=chl.CHL_FLAG_PARENTS),
     None),
    # smaller Common Label Tables (the tuner's candidates; the label table
    # holds the hubs left out)
    (dict(switch_ratio=1e6, common_hubs=8), None),
    (dict(switch_ratio=1e6, common_hubs=4, small_tree_expansions=NEVER_SMALL), None),
    # both switches with the other block sizes and bucket widths
    (dict(threads_per_tree=256, switch_ratio=1e6, small_tree_expansions=ALWAYS_SMALL,
          pruned_bucket_delta=1), None),
    (dict(threads_per_tree=512, psi_threshold=4.0, small_tree_expansions=512, bucket_delta=2), None),
]


@pytest.mark.parametrize("opts,check", SWEEP, ids=[",".join(f"{k}={v}" for k, v in o.items()) or "default"
                                                    for o, _ in SWEEP])
def test_switch_sweep_is_exact(family, opts, check):
    name, g, rank, ref, G, R = family
    L = chl.build_labels(G, R, **opts)
    st = L.stats()
    assert st["phases"] > 1, st
    assert st["small_tree_phases"] <= st["label_table_phases"], st
    if check is not None:
        assert check(st), (opts, st)
    assert_same(ref, *L.to_numpy())
    L.free()


def test_tuned_switch_points_are_exact(family):
    """chl_tune settles the switch points by whole builds; what it picks
    builds the canonical labels."""
    name, g, rank, ref, G, R = family
    opts, rep = chl.tune(G, R)
    assert rep["trials"] >= 3
    for k in ("switch_ratio", "small_tree_expansions", "big_tree_bucket_delta", "common_hubs"):
        assert k not in opts or opts[k] != 0
    L = chl.build_labels(G, R, **opts)
    assert_same(ref, *L.to_numpy())
    pairs = W.query_pairs(g, 20_000, seed=21)
    got = L.query(dev(pairs)).cpu().numpy().view(np.uint32)
    assert np.array_equal(got, O.query(ref, rank, pairs, threads=8))
    L.free()


@pytest.mark.parametrize("kind,first,later", [("random", False, True), ("scale-free", False, False)])
def test_narrow_width_after_big_pruned_trees(kind, first, later, capfd, monkeypatch):
    """Small graphs take the narrow width once a label-pruned phase's trees expanded
    as many vertices as there are (random graphs), not after the unpruned first phase."""
    rng = np.random.default_rng(2)
    if kind == "random":
        a, b = rng.integers(0, 4000, (2, 80_000))
        on = a != b
        key = np.unique(np.minimum(a, b)[on] * 4000 + np.maximum(a, b)[on])
        g = graph_of(4000, key // 4000, key % 4000, rng.integers(1, 101, len(key)))
        rank = W.degree_rank(g)
    else:
        g, rank = W.load("ba2k")
    ref = O.build_labels(g, rank, "plant", threads=8)
    monkeypatch.setenv("CHL_TRACE", "1")
    capfd.readouterr()
    L = chl.build_labels(DG(g), dev(rank), switch_ratio=1e6, small_tree_expansions=NEVER_SMALL)
    narrow = [" narrow" in x for x in capfd.readouterr().err.splitlines() if "table 1" in x]
    assert narrow[0] == first and any(narrow[1:]) == later, narrow
    assert_same(ref, *L.to_numpy())


@pytest.mark.parametrize("kind", ["uniform", "log-uniform", "few heavy", "huge"])
def test_bucket_width_by_spread_of_the_weights(kind, capfd, monkeypatch):
    """The default width of an unpruned phase: from the mean weight and the vertex
    count, narrower for heavy-tailed weights (mean square above four squared means)."""
    rng = np.random.default_rng(3)
    n, m = 3000, 30_000
    u, v = rng.integers(0, n, (2, m))
    on = u != v
    key = np.unique(np.minimum(u, v)[on] * n + np.maximum(u, v)[on])
    m = len(key)
    w = {"uniform": rng.integers(1, 101, m), "log-uniform": np.exp(rng.random(m) * np.log(100_000)).astype(np.int64) + 1,
         "few heavy": np.where(rng.random(m) < 0.01, 100_000, rng.integers(1, 11, m)),
         "huge": np.where(rng.random(m) < 0.001, 2**30, rng.integers(1, 11, m))}[kind]
    g = graph_of(n, key // n, key % n, w)
    rank = W.degree_rank(g)
    mean, square = float(w.mean()), float((w.astype(np.float64) ** 2).mean())
    want = mean / 128 if square > 4 * mean * mean else max(mean / 64, 1400 * mean / n)
    assert (square > 4 * mean * mean) == (kind != "uniform")
    width = 1
    while width * 1.5 < want:
        width *= 2
    monkeypatch.setenv("CHL_TRACE", "1")
    capfd.readouterr()
    L = chl.build_labels(DG(g), dev(rank))
    assert int(re.search(r" width (\d+) ", capfd.readouterr().err).group(1)) == width
    assert_same(O.build_labels(g, rank, "plant", threads=8), *L.to_numpy())


def line_before_scale_free(n, line, wave):
    """Pairs of vertices at the first 2 * wave positions, among them (in the second
    wave) the head of a long path; then a scale-free graph of n vertices; the rest
    of the path last. The path's tree is the long tail of the second phase, and the
    next phase's first trees label nearly n vertices each."""
    rng = np.random.default_rng(8)
    ba = W.barabasi_albert(n, 5, seed=8, wlo=1, whi=100)
    u, v, w = ba.edges()
    pairs = 2 * np.arange(wave)
    at = n + 2 * wave
    head = n + wave + wave // 2
    path = np.concatenate([[head], at + np.arange(line)])
    a = np.concatenate([u, n + pairs, path[:-1]]).astype(np.int64)
    b = np.concatenate([v, n + pairs + 1, path[1:]]).astype(np.int64)
    g = graph_of(at + line, a, b, np.concatenate([w, rng.integers(1, 100, wave + line)]).astype(np.int64))
    pos = np.empty(g.n, np.int64)
    pos[n:at] = np.arange(2 * wave)
    pos[:n] = 2 * wave + (n - 1 - W.degree_rank(ba).astype(np.int64))
    pos[at:] = at + np.arange(line)
    return g, (g.n - 1 - pos).astype(np.uint32)


@pytest.fixture(scope="module")
def long_tail():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g, rank = line_before_scale_free(33_000, 3000, sms)
    return g, rank, O.build_labels(g, rank, "plant", threads=8)


@pytest.mark.parametrize("opts", [dict(), dict(flags=chl.CHL_FLAG_PARENTS), dict(label_capacity=1000)],
                         ids=["default", "parents", "full buffer"])
def test_overlapped_trees(long_tail, opts, capfd, monkeypatch):
    """The next phase's first trees in a phase's tail, on a graph large enough for
    them by default; with a small label buffer they overflow theirs and are built
    again by their own phase."""
    g, rank, ref = long_tail
    monkeypatch.setenv("CHL_TRACE", "1")
    capfd.readouterr()
    L = chl.build_labels(DG(g), dev(rank), switch_ratio=1e6, **opts)
    err = capfd.readouterr().err
    if "label_capacity" in opts:
        assert any(int(x) for x in re.findall(r"(\d+) overlapped ones did not fit", err)), err
    else:
        assert L.stats()["overlapped_trees"] > 0, err
    assert_same(ref, *L.to_numpy())

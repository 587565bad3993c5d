"""Queries from several host threads, each on a stream of its own: more callers
at once than the library has staging blocks, in every mode, host and device
pairs, good and bad ones, against the oracle; and short queries beside a long
kernel of another stream. Integers: comparisons are exact."""
import threading
import time

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


@pytest.fixture(scope="module")
def held():
    g = W.barabasi_albert(3000, 4, seed=6, wlo=1, whi=100)
    rank = W.degree_rank(g)
    L = chl.build_labels(DG(g), dev(rank), flags=chl.CHL_FLAG_PARENTS)
    parts = [chl.build_labels(DG(g), dev(rank), root_begin=a, root_end=b) for a, b in ((0, 40), (40, g.n))]
    return g, rank, L, parts, O.build_labels(g, rank, "plant", threads=8)


def in_threads(n, f):
    """Runs f(0) .. f(n - 1) in threads of their own; raises what one of them raised."""
    err = []

    def body(i):
        try:
            f(i)
        except BaseException as e:
            err.append(e)

    ts = [threading.Thread(target=body, args=(i,)) for i in range(n)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if err:
        raise err[0]


def test_many_callers_in_every_mode(held):
    g, rank, L, parts, ref = held
    n = 14
    start = threading.Barrier(n)
    pairs = [np.random.default_rng(i).integers(0, g.n, (1 + 37 * i, 2)).astype(np.uint32) for i in range(n)]
    want = [O.query(ref, rank, p) for p in pairs]
    bad = np.array([[0, g.n]], np.uint32)

    def caller(i):
        torch.cuda.set_device(0)
        s = torch.cuda.Stream()
        ask = [lambda p: L.query(p, stream=s.cuda_stream),
               lambda p: L.query(p, stream=s.cuda_stream, grouped=True),
               lambda p: chl.query_partitioned(parts, p, stream=s.cuda_stream)]
        on_dev = dev(pairs[i])
        torch.cuda.synchronize()
        start.wait()
        for k in range(30):
            with torch.cuda.stream(s):
                torch.cuda._sleep(200_000)  # the call holds its block while its stream is busy
            f = ask[(i + k) % 3]
            if k % 10 == 9:
                with pytest.raises(chl.ChlError, match="vertex id"):
                    f(bad)
            got = f(pairs[i]) if k % 2 else f(on_dev).cpu().numpy().view(np.uint32)
            assert np.array_equal(got, want[i])
        paths, lens = L.paths(pairs[i][:20], max_len=8, stream=s.cuda_stream)
        assert ((lens >= 1) == (want[i][:20] != 0xFFFFFFFF)).all() and (paths[:, 0] == pairs[i][:20, 0]).all()

    in_threads(n, caller)


def test_calls_do_not_wait_for_another_stream(held):
    """Six calls in flight at once end while a kernel of another stream runs on."""
    g, rank, L, parts, ref = held
    n = 6
    pairs = np.random.default_rng(3).integers(0, g.n, (5, 2)).astype(np.uint32)
    want = O.query(ref, rank, pairs)
    other, streams = torch.cuda.Stream(), [torch.cuda.Stream() for _ in range(n)]
    in_threads(n, lambda i: L.query(pairs, stream=streams[i].cuda_stream))  # warm
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    torch.cuda._sleep(20_000_000)
    t1.record()
    torch.cuda.synchronize()
    per_ms = 20_000_000 / t0.elapsed_time(t1)
    with torch.cuda.stream(other):
        torch.cuda._sleep(int(per_ms * 1500))
    took = [0.0] * n

    def caller(i):
        for _ in range(3):
            with torch.cuda.stream(streams[i]):
                torch.cuda._sleep(int(per_ms * 20))
            a = time.perf_counter()
            got = L.query(pairs, stream=streams[i].cuda_stream)
            took[i] = max(took[i], time.perf_counter() - a)
            assert np.array_equal(got, want)

    in_threads(n, caller)
    still = not other.query()
    torch.cuda.synchronize()
    assert still and max(took) < 0.7, (took, still)


"""Label tables of the label-pruned phases in both entry forms (one word where
hub positions and distances fit 32 bits together, else two), the change from
one to the other as the table grows, and the Common Label Table's comparison at
the ends of its range, against the oracle. Integers: comparisons are exact."""
import pytest

import oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1907_00140_gb300 as chl  # noqa: E402
from test_gpu_parity import DG, dev, assert_same  # noqa: E402


# weights up to: always packed; packed until the table's hubs need the bits;
# never packed (distances past 24 bits); 8-byte keys and distances near 2^32
@pytest.mark.parametrize("whi", [100, 60_000, 6_000_000, 150_000_000])
@pytest.mark.parametrize("opts", [dict(), dict(flags=chl.CHL_FLAG_DENSE_ROOT_LABELS), dict(query_stage_kb=8),
                                  dict(flags=chl.CHL_FLAG_PARENTS), dict(common_hubs=7, threads_per_tree=64)],
                         ids=["default", "dense", "staged", "parents", "7 hubs"])
def test_table_forms(whi, opts):
    g = W.barabasi_albert(12000, 4, seed=6, wlo=max(1, whi // 50), whi=whi)
    rank = W.degree_rank(g)
    ref = O.build_labels(g, rank, "pll")
    assert int(ref.dist.max()) > 2 * (whi // 50)
    L = chl.build_labels(DG(g), dev(rank), **opts)
    assert L.stats()["label_table_phases"] > 2
    assert_same(ref, *L.to_numpy())

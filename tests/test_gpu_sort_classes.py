"""The label sort at the edges of its length classes (32, 128, 256, 512 and
1,024 labels sorted by one warp, longer lists by a block): the lists of two
centres are one label short of an edge, at it or past it, against the oracle.
Integers: comparisons are exact."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import assert_same, gpu_labels  # noqa: E402
from test_gpu_query_blocks import two_centres  # noqa: E402


@pytest.mark.parametrize("length", [2, 32, 33, 127, 128, 129, 256, 257, 511, 512, 513, 1024, 1025])
def test_lists_at_the_edges_of_the_sort(length):
    g, rank, _ = two_centres(length - 1, 1, seed=length)
    ref = O.build_labels(g, rank, "plant", threads=8)
    assert np.diff(np.asarray(ref.offsets).astype(np.int64))[:2].tolist() == [length, length]
    assert_same(ref, *gpu_labels(g, rank)[1:4])

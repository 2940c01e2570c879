"""Priority range search at the edges of its box hierarchy and id buffers:
point counts around 32, 1024 and 32768 (one, two, three levels), ids asked for
around the buffer sizes and the one-pass limit of 512, ids that fall along the
key order (every match improves on the buffer), and ragged batches whose
upper-level nodes straddle instances.  Exact, as the oracle."""
import numpy as np
import pytest

import workloads as W
from test_gpu_range import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1023, 1024, 1025, 32768, 33000])
def test_sizes_around_the_levels(n):
    rng = np.random.default_rng(n)
    pts = W.random_blobs(n, 3, 40) if n > 40 else rng.random((n, 3)).astype(np.float32)
    check([pts], [3], [rng.integers(1, 30, n).astype(np.int32)], 64, 7, 5)


@pytest.mark.parametrize("max_out", [1, 32, 33, 64, 512, 513])
def test_ids_around_the_buffers(max_out):
    rng = np.random.default_rng(6)
    pts = W.random_blobs(9000, 2, 41)
    check([pts], [2], [rng.integers(-5, 5, 9000).astype(np.int32)], 80, max_out, 6)


def test_ids_descending_along_the_key_order():
    pts = np.arange(5000, dtype=np.int32)[::-1].reshape(-1, 1).copy()
    check([pts], [1], [np.full(5000, 3, np.int32)], 48, 16, 7, dtype=np.int32)


def test_nodes_straddling_instances():
    rng = np.random.default_rng(8)
    sizes = [int(x) for x in rng.integers(1, 90, 120)] + [2500, 40]
    dims = [2] * len(sizes)
    insts = [W.random_blobs(n, 2, 700 + i) for i, n in enumerate(sizes)]
    check(insts, dims, [rng.integers(1, 9, n).astype(np.int32) for n in sizes], 300, 20, 9)

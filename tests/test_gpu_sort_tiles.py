"""Point counts around the radix sort's changes of tile size (2^17 and 2^21
points) and of the density's chunk split, against the kd-tree oracle; and the
64-bit integer densities of int32 points in the binary64 mode at the largest
coordinates the library accepts.  Exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_2305_11335_gb300 as dpc
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16385, 38912, 131071, 131073, 2097152, 2097153])
def test_sizes_around_the_tiles(n):
    pts = W.random_blobs(n, 2, 17, dtype=np.int32, scale=5e5 if n < 1 << 20 else 4e6)
    dc = 900.0
    ref = oracle.tree_run(pts, [dc])
    out = {k: v[0].cpu().numpy() for k, v in dpc.run(torch.from_numpy(pts).cuda(), [dc], 2, 3, 5e3).items()}
    for k in ("rho", "lam", "delta"):
        assert np.array_equal(out[k].view(np.int64) if k == "delta" else out[k],
                              ref[k][0].view(np.int64) if k == "delta" else ref[k][0]), k


@pytest.mark.parametrize("d", [1, 2, 3, 5, 8])
def test_integer_densities_at_the_largest_coordinates(d):
    rng = np.random.default_rng(d)
    pts = rng.choice(np.array([-(1 << 24), -(1 << 24) + 1, 0, 3, (1 << 24) - 1, 1 << 24]), (5000, d)).astype(np.int32)
    t = torch.from_numpy(pts).cuda()
    for dc in (0.0, 1.0, float(1 << 24), 2.0 ** 25 * d ** 0.5, 1e12):
        want = oracle.density(pts, dc)
        got = dpc.dpc_density(t, dpc.Batch.single(5000, d, [dc]), precision="fp64", sync=True)[0].cpu().numpy()
        assert np.array_equal(got, want), dc

"""Cutoffs and coordinates at the top of the accepted range, against the
oracle, for sets above the all-pairs limits whose sizes leave the last tile
partly empty: a padding candidate must never count, however large the cutoff.
One cutoff and sweeps of one to four cutoffs per grid level, the tensor tiles
of 5 to 8 dimensions and the allocation-free density.  Exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_2305_11335_gb300 as dpc
from _gpu_util import parity

pytestmark = pytest.mark.gpu


def densities(pts, cuts, **kw):
    t = torch.from_numpy(pts).cuda()
    batch = dpc.Batch.single(len(pts), pts.shape[1], cuts)
    return dpc.dpc_density(t, batch, sync=True, **kw).cpu().numpy()


def far_blobs(n, d, center, spread, seed):
    """Blobs around +-center: every distance is a small multiple of `spread`
    within a blob, about 2 center between blobs."""
    rng = np.random.default_rng(seed)
    c = center * rng.choice([-1.0, 1.0], (4, d))
    return (c[rng.integers(0, 4, n)] + rng.normal(0.0, spread, (n, d))).astype(np.float32)


@pytest.mark.parametrize("d", [5, 6, 7, 8])
@pytest.mark.parametrize("layout", ["auto", "tensor"])
def test_tensor_tiles_everything_within_the_cutoff(d, layout):
    n = 17009
    pts = np.random.default_rng(d).random((n, d), dtype=np.float32)
    for cuts in ([1e16], [1e20], [1e16, 1.5e16, 1.9e16, 1e15, 0.2]):
        got = densities(pts, cuts, layout=layout)
        for c, dc in enumerate(cuts):
            want = oracle.density(pts, dc) if dc < 10.0 else np.full(n, n)
            assert np.array_equal(got[c], want), (cuts, c)


@pytest.mark.parametrize("d", [5, 8])
@pytest.mark.parametrize("center,spread", [(1e17, 1e15), (1e18, 2e16)])
def test_tensor_tiles_far_coordinates(d, center, spread):
    pts = far_blobs(9013, d, center, spread, d)
    for cuts in ([2.0 * spread], [2.0 * spread, 2.5 * spread, 3.0 * spread, 2.2 * spread]):
        parity(pts, cuts, rho_noise=3, rho_min=50, delta_min=4.0 * spread)


def test_static_density_in_tensor_tiles():
    for n, dc in ((20000, 1e16), (20011, 1e16), (20011, 1e20)):
        pts = np.random.default_rng(n).random((n, 7), dtype=np.float32)
        got = dpc.dpc_density_static(torch.from_numpy(pts).cuda(), dc, sync=True).cpu().numpy()
        assert (got == n).all(), (n, dc)


CUTS = [1e18, 1e20, 1e200, 1.7e308]  # squares beyond 2^122, past float32, past binary64


@pytest.mark.parametrize("d", [1, 2, 3, 4, 7])
@pytest.mark.parametrize("dtype", [np.float32, np.int32])
def test_segments_everything_within_the_cutoff(d, dtype):
    n = 17003
    rng = np.random.default_rng(40 + d)
    pts = rng.random((n, d), dtype=np.float32) if dtype == np.float32 else rng.integers(0, 1000, (n, d), dtype=np.int32)
    small = 0.05 if dtype == np.float32 else 30.0
    want = oracle.density(pts, small)
    for prec in ("fp32", "fp64"):
        for layout in ("auto", "segment"):
            for cuts in [[c] for c in CUTS] + [CUTS, [1e200, 1.1e200, small], [1e20, 1.1e20, 1.2e20, 1.3e20, 1.4e20]]:
                got = densities(pts, cuts, precision=prec, layout=layout)
                for c, dc in enumerate(cuts):
                    assert np.array_equal(got[c], want if dc == small else np.full(n, n)), (prec, layout, cuts, c)


def test_segments_count_no_band_pairs_beyond_float32():
    """Every squared distance is finite in float32, so none is undecided by a
    filter whose outer threshold is infinite."""
    pts = np.random.default_rng(3).random((17003, 3), dtype=np.float32)
    for cuts in ([1e20], [1e20, 1.1e20]):
        densities(pts, cuts)
        assert dpc.dpc_get_stats()["band_pairs"] == 0, cuts


@pytest.mark.parametrize("d", [2, 3])
def test_run_with_an_infinite_square(d):
    pts = np.random.default_rng(50 + d).random((17003, d), dtype=np.float32)
    parity(pts, [1e200, 1e199, 0.03], rho_noise=2, rho_min=5, delta_min=0.1)


@pytest.mark.parametrize("layout", ["union", "pairs", "cell"])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 7])
def test_other_layouts_everything_within_the_cutoff(d, layout):
    n = 1003 if layout == "cell" else 5003
    rng = np.random.default_rng(60 + d)
    for pts in (rng.random((n, d), dtype=np.float32), rng.integers(0, 1000, (n, d), dtype=np.int32)):
        for prec in ("fp32", "fp64"):
            for cut in CUTS:
                got = densities(pts, [cut], precision=prec, layout=layout)
                assert (got[0] == n).all(), (prec, cut)

"""The edge cases of the parity tests at sizes above the all-pairs limits, so
that the grid, the tree search and the sweeps meet them too: pairs at the
cutoff and a float step beside it, large offsets with tiny spreads, integer
ties, zero and huge cutoffs, sets of equal points.  Exact."""
import numpy as np
import pytest

import workloads as W
from _gpu_util import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [2, 3, 5])
def test_boundary_band(d):
    rng = np.random.default_rng(5 + d)
    m = 8600
    base = rng.random((m, d)) * 60.0
    dc = 0.37
    u = rng.standard_normal((m, d))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    pts = np.concatenate([base, base + dc * u]).astype(np.float32)
    for step in range(2):  # partners nudged by float steps in random directions
        k = rng.integers(-1, 2, (m, d))
        part = pts[m:]
        pts[m:] = np.where(k == 0, part, np.nextafter(part, np.where(k < 0, -np.inf, np.inf).astype(np.float32)))
    parity(pts, [dc], rho_noise=1, rho_min=2, delta_min=1.0)
    parity(pts, [dc, 0.4], rho_noise=1, rho_min=2, delta_min=1.0)


@pytest.mark.parametrize("d", [2, 6])
def test_large_offset_cancellation(d):
    rng = np.random.default_rng(9 + d)
    pts = (1e5 + rng.random((17001, d)) * 0.9).astype(np.float32)
    for cuts in ([0.01], [0.01, 0.003, 0.011], [0.2]):
        parity(pts, cuts, rho_noise=1, rho_min=2, delta_min=0.05)


@pytest.mark.parametrize("d,extent", [(2, 70), (3, 17)])
def test_equidistant_ties_int(d, extent):
    pts = np.random.default_rng(3).integers(0, extent, (17000, d)).astype(np.int32)
    for cuts in ([2.0], [1.0, 2.0, 2.5]):
        parity(pts, cuts, rho_noise=2, rho_min=4, delta_min=3.0)


@pytest.mark.parametrize("cuts", [[0.0], [1e-6], [50.0], [0.0, 1e-6, 50.0]])
def test_zero_and_huge_cutoff(cuts):
    pts = W.random_blobs(17000, 2, 31, dtype=np.float32, dup_frac=0.05)
    parity(pts, cuts, rho_noise=1, rho_min=2, delta_min=0.05)


@pytest.mark.parametrize("d", [3, 8])
def test_all_equal(d):
    pts = W.all_equal(8301, d)
    for cuts in ([0.0], [0.0, 1.0]):
        parity(pts, cuts, rho_noise=1, rho_min=1, delta_min=0.5)

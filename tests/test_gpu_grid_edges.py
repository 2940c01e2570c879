"""The edge cases of the parity tests at sizes above the all-pairs limits, so
that the grid, the tree search and the sweeps meet them too: pairs at the
cutoff and a float step beside it, large offsets with tiny spreads, integer
ties, zero and huge cutoffs, sets of equal points, the entry points one by one
with densities of no cutoff, bad coordinates.  Exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_2305_11335_gb300 as dpc
import workloads as W
from _gpu_util import assert_same, bits, parity

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


@pytest.mark.parametrize("d", [1, 2, 3, 5, 8])
def test_split_entry_points_and_any_rho(d):
    """dpc_dependent is a function of (points, rho): the densities of the
    cutoff, then seeded random ones (zero among them) with a noise skip."""
    n = 17003
    pts = W.random_blobs(n, d, 55 + d, dup_frac=0.01)
    dc = 0.01 * d if d < 5 else 0.04 * d
    t = torch.from_numpy(pts).cuda()
    batch = dpc.Batch.single(n, d, [dc])
    params = dpc.make_params(batch, 3, 6, 0.2)
    ref = oracle.run(pts, dc, 3, 6, 0.2)
    rho = dpc.dpc_density(t, batch, sync=True)[0].contiguous()
    lam, delta = dpc.dpc_dependent(t, batch, 0, rho, sync=True)
    label = dpc.dpc_cluster(batch, 0, params, rho, lam, delta, sync=True)
    assert_same({"rho": rho.cpu().numpy(), "lam": lam.cpu().numpy(), "delta": delta.cpu().numpy(),
                 "label": label.cpu().numpy()}, ref)
    any_rho = np.random.default_rng(d).integers(0, 40, n).astype(np.int32)
    for skip in (0, 3):
        rl, rd = oracle.dependent(pts, any_rho, rho_skip=skip)
        for prec in ("fp32", "fp64"):
            lam, delta = dpc.dpc_dependent(t, batch, 0, torch.from_numpy(any_rho).cuda(), rho_skip=skip,
                                           precision=prec, sync=True)
            assert np.array_equal(lam.cpu().numpy(), rl), (skip, prec)
            assert np.array_equal(bits(delta.cpu().numpy()), bits(rd)), (skip, prec)


@pytest.mark.parametrize("d", [1, 2, 7])
def test_bad_coordinates_reported(d):
    """On the grid and in its sweeps; the library recovers."""
    good = W.random_blobs(17000, d, 4)
    for bad in (np.nan, np.inf, 1.2e18):
        pts = good.copy()
        pts[9001, d - 1] = bad
        for cuts in ([0.05], [0.05, 0.06]):
            with pytest.raises(dpc.DpcError) as e:
                dpc.run(torch.from_numpy(pts).cuda(), cuts, 1, 1, 1.0)
            assert e.value.code == dpc.DPC_ERR_DATA
    parity(good[:9000], [0.02 * d], precisions=("fp32",))

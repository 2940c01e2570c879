"""Small instances (all pairs, no grid; one-launch labels) against the oracle:
sizes around a warp, a CTA's step of 256 candidates and the limits of the
rule, every dimension, both precisions, integer ties (the binary64 ranking),
batches of one and of mixed dimensions, more cutoffs than kernel arguments
hold, the allocation-free density and label cycles.  Exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_2305_11335_gb300 as dpc
import workloads as W
from _gpu_util import assert_same, parity
from test_gpu_batch import check_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", range(1, 9))
@pytest.mark.parametrize("n", [1, 7, 33, 257, 1000])
def test_every_dimension(n, d):
    pts = W.random_blobs(n, d, 800 + n + d, dup_frac=0.02) if n > 40 else np.random.default_rng(n + d).random(
        (n, d)).astype(np.float32)
    parity(pts, [0.05 * d, 0.1 * d], rho_noise=2, rho_min=4, delta_min=0.2)


@pytest.mark.parametrize("n", [2048, 2049, 4096, 4097, 8192, 8193, 16384, 16385])
def test_sizes_around_the_limits(n):
    pts = W.random_blobs(n, 2, 820)
    parity(pts, [0.02])
    t = torch.from_numpy(pts).cuda()
    want = oracle.density(pts, 0.02)
    for prec in ("fp32", "fp64"):
        got = dpc.dpc_density(t, dpc.Batch.single(n, 2, [0.02, 0.03]), precision=prec, sync=True)
        assert np.array_equal(got[0].cpu().numpy(), want)
        assert np.array_equal(got[1].cpu().numpy(), oracle.density(pts, 0.03))
        assert np.array_equal(dpc.dpc_density_static(t, 0.02, precision=prec, sync=True).cpu().numpy(), want)


def test_integer_ties_and_skipped_points():
    pts = np.random.default_rng(5).integers(0, 24, (3000, 2)).astype(np.int32)
    parity(pts, [0.0, 1.0, 2.0, 5.0], rho_noise=3, rho_min=6, delta_min=1.0)
    t = torch.from_numpy(pts).cuda()
    out = dpc.run(t, [2.0], 30, 40, 1.0, skip_noise=True)
    ref = oracle.run(pts, 2.0, 30, 40, 1.0, rho_skip=30)
    assert_same({k: v[0].cpu().numpy() for k, v in out.items()}, ref)


@pytest.mark.parametrize("dims", [[3], [5, 6, 8]])
def test_batches(dims):
    sizes = [0, 1, 2, 31, 32, 33, 700, 1500, 64]
    ds = [dims[i % len(dims)] for i in range(len(sizes))]
    insts = [W.random_blobs(n, d, 830 + i) if n > 40 else np.random.default_rng(i).random((n, d)).astype(np.float32)
             for i, (n, d) in enumerate(zip(sizes, ds))]
    check_run(sizes, ds, insts, [[0.1, 0.15, 0.2] for _ in sizes], np.float32, "fp32", 31)


def test_more_cutoffs_than_kernel_arguments():
    pts = W.random_blobs(900, 3, 840)
    parity(pts, [0.02 * 1.1 ** k for k in range(19)], precisions=("fp32",))


def test_bad_coordinates_are_reported():
    pts = W.random_blobs(500, 3, 841)
    pts[499, 2] = np.nan
    with pytest.raises(dpc.DpcError) as e:
        dpc.run(torch.from_numpy(pts).cuda(), [0.1], 2, 3, 0.1)
    assert e.value.code == dpc.DPC_ERR_DATA
    with pytest.raises(dpc.DpcError) as e:
        dpc.dpc_density_static(torch.full((40, 2), 1 << 25, dtype=torch.int32).cuda(), 1.0, sync=True)
    assert e.value.code == dpc.DPC_ERR_DATA


@pytest.mark.parametrize("n", [3, 5000, 32768, 32769])
def test_label_chains_and_cycles(n):
    """One chain through every point, then the same closed to a cycle of the
    whole set and of two points with everything leading into it."""
    batch = dpc.Batch.single(n, 2, [1.0])
    params = dpc.make_params(batch, 0, 1, 1e9)
    perm = np.random.default_rng(n).permutation(n)
    lam = np.empty(n, np.int32)
    lam[perm[1:]] = perm[:-1]
    lam[perm[0]] = -1
    rho = torch.ones(n, dtype=torch.int32).cuda()
    delta = torch.zeros(n, dtype=torch.float64).cuda()
    got = dpc.dpc_cluster(batch, 0, params, rho, torch.from_numpy(lam).cuda(), delta, sync=True)
    assert (got.cpu().numpy() == perm[0]).all()
    for last in (perm[-1], perm[1]):
        lam[perm[0]] = last
        with pytest.raises(dpc.DpcError) as e:
            dpc.dpc_cluster(batch, 0, params, rho, torch.from_numpy(lam).cuda(), delta, sync=True)
        assert e.value.code == dpc.DPC_ERR_DATA

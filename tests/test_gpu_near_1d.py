"""The 1-D near phase on both sides of its rule (block scan on dense cells, tree
search elsewhere), alone and in sweeps, single sets and batches, both
precisions, with ties and skipped points.  Exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_2305_11335_gb300 as dpc
import workloads as W
from _gpu_util import assert_same

pytestmark = pytest.mark.gpu


def reference(pts, cuts, noise, rho_min, delta_min, skip=0):
    o = oracle.tree_run(pts, cuts, rho_skip=skip)
    return [{"rho": o["rho"][c], "lam": o["lam"][c], "delta": o["delta"][c],
             "label": oracle.cluster(o["rho"][c], o["lam"][c], o["delta"][c], noise, rho_min, delta_min)}
            for c in range(len(cuts))]


@pytest.mark.parametrize("n,r,prec,near", [(131072, 0.05, "fp32", 1), (131073, 0.05, "fp32", 1), (131071, 0.05, "fp32", 3),
                                           (140000, 0.00002, "fp32", 3), (140000, 0.05, "fp64", 3)])
def test_dense_and_sparse_cells(n, r, prec, near):
    """Against the kd-tree oracle."""
    pts = W.random_blobs(n, 1, 3, dup_frac=0.001)
    for cuts in ([r], [r, 1.05 * r]):
        batch = dpc.Batch.single(n, 1, cuts)
        t = torch.from_numpy(pts).cuda()
        out = dpc.dpc_run(t, batch, dpc.make_params(batch, 3, 20, 0.01), precision=prec, sync=True)
        assert dpc.dpc_get_stats()["near_layout"] == near
        for c, ref in enumerate(reference(pts, cuts, 3, 20, 0.01)):
            assert_same({k: v[c].cpu().numpy() for k, v in out.items()}, ref, "%s %d" % (prec, c))


def test_skipped_points():
    n = 140000
    pts = W.random_blobs(n, 1, 5)
    batch = dpc.Batch.single(n, 1, [0.05])
    out = dpc.dpc_run(torch.from_numpy(pts).cuda(), batch, dpc.make_params(batch, 4000, 9000, 0.01), skip_noise=True,
                      sync=True)
    assert dpc.dpc_get_stats()["near_layout"] == 1
    assert_same({k: v[0].cpu().numpy() for k, v in out.items()}, reference(pts, [0.05], 4000, 9000, 0.01, 4000)[0])


def test_integer_ties():
    pts = np.random.default_rng(4).integers(0, 3000, (132000, 1)).astype(np.int32)
    batch = dpc.Batch.single(len(pts), 1, [40.0])
    out = dpc.dpc_run(torch.from_numpy(pts).cuda(), batch, dpc.make_params(batch, 3, 20, 2.0), sync=True)
    assert dpc.dpc_get_stats()["near_layout"] == 1
    assert_same({k: v[0].cpu().numpy() for k, v in out.items()}, reference(pts, [40.0], 3, 20, 2.0)[0])


def test_batch_of_dense_and_sparse_instances():
    insts = [W.random_blobs(n, 1, 30 + n) for n in (70000, 40, 62000)] + [np.zeros((1, 1), np.float32)]
    sizes = [len(p) for p in insts]
    cuts = [[0.1], [0.1], [0.0001], [0.1]]
    batch = dpc.Batch.packed(sizes, [1] * 4, cuts)
    flat = torch.from_numpy(np.concatenate([p.reshape(-1) for p in insts])).cuda()
    out = dpc.dpc_run(flat, batch, dpc.make_params(batch, 3, 20, 0.01), sync=True)
    for i, p in enumerate(insts):
        lo, hi = batch.pt_offset[i], batch.pt_offset[i + 1]
        assert_same({k: v[0, lo:hi].cpu().numpy() for k, v in out.items()}, reference(p, cuts[i], 3, 20, 0.01)[0], str(i))

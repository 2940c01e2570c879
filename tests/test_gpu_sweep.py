"""Cutoff sweeps (cutoffs that share cells counted in one pass, the near phase
on a smaller cutoff's cells) against the oracle: one to five cutoffs per grid
level, unsorted and repeated cutoffs, zero among them, ratios beyond the near
phase's three levels, instances whose sweeps disagree about the order, every
gridded dimension, both precisions, and the tensor tiles on sparse and dense
cells.  Exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_2305_11335_gb300 as dpc
import workloads as W
from _gpu_util import assert_same

pytestmark = pytest.mark.gpu


def check(insts, cuts, prec="fp32", skip=False, dtype=np.float32):
    sizes, dims = [len(p) for p in insts], [p.shape[1] for p in insts]
    batch = dpc.Batch.packed(sizes, dims, cuts)
    params = dpc.make_params(batch, 3, 5, 0.3)
    flat = torch.from_numpy(np.concatenate([p.reshape(-1) for p in insts]).astype(dtype)).cuda()
    out = {k: v.cpu().numpy() for k, v in dpc.dpc_run(flat, batch, params, precision=prec, sync=True,
                                                      skip_noise=skip).items()}
    den = dpc.dpc_density(flat, batch, precision=prec, sync=True).cpu().numpy()
    for i, p in enumerate(insts):
        lo, hi = batch.pt_offset[i], batch.pt_offset[i + 1]
        for c, dc in enumerate(cuts[i]):
            ref = oracle.run(p.astype(dtype), dc, 3, 5, 0.3, rho_skip=3 if skip else 0)
            assert_same({k: v[c, lo:hi] for k, v in out.items()}, ref, "%s inst %d cut %d" % (prec, i, c))
            assert np.array_equal(den[c, lo:hi], ref["rho"])


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 6, 7, 8])
def test_levels_and_group_sizes(d, prec):
    n = 17000 if prec == "fp32" and d < 6 else 9000
    pts = W.random_blobs(n, d, 60 + d, dup_frac=0.01)
    d0 = 0.003 * d if d <= 4 else 0.02 * d
    check([pts], [[d0 * 1.7, d0, d0 * 1.1, d0 * 2.0, d0 * 1.3, d0 * 1.5, d0 * 1.9, d0 * 3.0]], prec)


def test_zero_repeated_and_distant_cutoffs():
    pts = W.random_blobs(17000, 2, 71, dup_frac=0.05)
    check([pts], [[0.004, 0.0, 0.004, 0.2]])
    check([pts], [[0.001, 0.05, 0.3, 0.0011]])
    ip = np.random.default_rng(2).integers(0, 60, (17000, 3)).astype(np.int32)
    check([ip], [[1.0, 2.0, np.sqrt(3.0), 4.0]], dtype=np.int32, skip=True)


def test_instances_disagree_about_the_order():
    insts = [W.random_blobs(n, d, 80 + n) for n, d in ((17000, 3), (40, 3), (9000, 7), (300, 5), (17500, 2), (1, 2))]
    cuts = [[0.01, 0.02, 0.03], [0.5, 0.1, 0.2], [0.3, 0.1, 0.11], [0.1, 0.4, 0.3], [0.02, 0.005, 0.011],
            [1.0, 0.0, 2.0]]
    check(insts, cuts)


@pytest.mark.parametrize("d", [5, 8])
def test_tensor_tiles_sparse_and_dense_cells(d):
    rng = np.random.default_rng(d)
    dense = np.concatenate([rng.normal(0.5, 0.004, (7000, d)), rng.random((5000, d))]).astype(np.float32)
    check([dense], [[0.02, 0.024, 0.05]])
    lattice = rng.integers(0, 3, (9000, d)).astype(np.int32)  # every distance an integer square: the band and its recount
    check([lattice], [[1.0, np.sqrt(2.0), 2.0]], dtype=np.int32)

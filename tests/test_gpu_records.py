"""The far search on trees deeper than its shared-memory stack, and classes of
5- and 6-dimensional points (child records of six coordinates) alone and beside
wider ones, against the brute-force oracle.  Exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_2305_11335_gb300 as dpc
import workloads as W
from _gpu_util import assert_same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("d", [2, 3])
def test_stack_beyond_shared_memory(d, prec):
    # 300 copies of the origin, 301 of 2^k on every axis: the search of the
    # highest copy of the origin, which has no bound from its sorted neighbours,
    # leaves a farther child behind on each of 21 d levels
    pts = [np.zeros((300, d), np.int32)]
    for k in range(21):
        for a in range(d):
            x = np.zeros((301, d), np.int32)
            x[:, a] = 1 << k
            pts.append(x)
    pts = np.concatenate(pts)
    dc = 0.5
    out = dpc.run(torch.from_numpy(pts).cuda(), [dc], 2, 3, 10.0, precision=prec)
    ref = oracle.run(pts, dc, 2, 3, 10.0)
    assert_same({k: v[0].cpu().numpy() for k, v in out.items()}, ref, "d %d %s" % (d, prec))


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("dims", [[5, 6, 5], [6], [5, 8], [7, 6]])
def test_record_dimensions(dims, prec):
    insts = [W.random_blobs(9000 + 31 * i, d, 40 + d, dup_frac=0.01) for i, d in enumerate(dims)]
    cuts = [[0.02 * d, 0.05 * d] for d in dims]
    batch = dpc.Batch.packed([len(p) for p in insts], dims, cuts)
    params = dpc.make_params(batch, 3, 5, 0.3)
    flat = torch.from_numpy(np.concatenate([p.reshape(-1) for p in insts])).cuda()
    out = {k: v.cpu().numpy() for k, v in dpc.dpc_run(flat, batch, params, precision=prec, sync=True).items()}
    for i, p in enumerate(insts):
        lo, hi = batch.pt_offset[i], batch.pt_offset[i + 1]
        for c, dc in enumerate(cuts[i]):
            assert_same({k: v[c, lo:hi] for k, v in out.items()}, oracle.run(p, dc, 3, 5, 0.3),
                        "%s inst %d cut %d" % (prec, i, c))

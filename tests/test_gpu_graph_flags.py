"""Captured calls that differ only in a flag must not replay each other's
graph: skip_noise changes lambda and delta of the noise points, the near
phase's level the kernels' arguments.  Below and above the all-pairs limit."""
import numpy as np
import pytest
import torch

import oracle
import paper_2305_11335_gb300 as dpc
import workloads as W
from _gpu_util import assert_same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [900, 9000])
@pytest.mark.parametrize("ncut", [1, 2])
def test_skip_noise_alternates(n, ncut):
    s = torch.cuda.Stream()
    pts = W.random_blobs(n, 2, 910 + n)
    cuts = [0.02, 0.03][:ncut]
    batch = dpc.Batch.single(n, 2, cuts)
    params = dpc.make_params(batch, 12, 20, 0.1)
    refs = {skip: [oracle.run(pts, dc, 12, 20, 0.1, rho_skip=12 if skip else 0) for dc in cuts]
            for skip in (False, True)}
    assert not np.array_equal(refs[False][0]["lam"], refs[True][0]["lam"])
    t = torch.from_numpy(pts).cuda()
    out = None
    torch.cuda.synchronize()
    for skip in (False, True, True, False, True):
        with torch.cuda.stream(s):
            out = dpc.dpc_run(t, batch, params, stream=s, out=out, graph=True, skip_noise=skip, sync=True)
        for c in range(ncut):
            assert_same({k: v[c].cpu().numpy() for k, v in out.items()}, refs[skip][c], "skip %s cut %d" % (skip, c))


def test_near_shift_alternates():
    s = torch.cuda.Stream()
    n = 9000
    pts = W.random_blobs(n, 2, 920)
    batch = dpc.Batch.single(n, 2, [0.02])
    params = dpc.make_params(batch, 3, 5, 0.1)
    ref = oracle.run(pts, 0.02, 3, 5, 0.1)
    t = torch.from_numpy(pts).cuda()
    out = None
    torch.cuda.synchronize()
    for shift in (0, 1, 0, 2):
        with torch.cuda.stream(s):
            out = dpc.dpc_run(t, batch, params, stream=s, out=out, graph=True, near_shift=shift, layout="segment",
                              sync=True)
        assert_same({k: v[0].cpu().numpy() for k, v in out.items()}, ref, "shift %d" % shift)
        assert dpc.dpc_get_stats(s)["near_shift"] == shift

"""More cutoffs than one grid dimension of a launch can count (65,535) on a
small set: every row of the result, against a sorted list of distances."""
import numpy as np
import pytest
import torch

import paper_2305_11335_gb300 as dpc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ncut", [65535, 65536, 131075])
def test_densities_of_many_cutoffs(ncut):
    pts = np.random.default_rng(5).integers(0, 900, (33, 2)).astype(np.int32)
    cuts = np.linspace(0.0, 1300.0, ncut)
    got = dpc.dpc_density(torch.from_numpy(pts).cuda(), dpc.Batch.single(33, 2, cuts.tolist()), sync=True).cpu().numpy()
    p = pts.astype(np.int64)
    s = ((p[:, None] - p[None]) ** 2).sum(-1).astype(np.float64)
    s.sort(axis=1)
    want = np.stack([np.searchsorted(s[i], cuts * cuts, side="right") for i in range(33)], axis=1)
    assert np.array_equal(got, want)

"""Binary64 sweeps whose levels hold four cutoffs and one over: the last one is
counted pair by pair on the group's cells.  Single instances, and a batch whose
instances disagree about which cutoff is the largest.  Exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_2305_11335_gb300 as dpc
import workloads as W
from test_gpu_sweep import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [1, 2, 3, 4, 6])
@pytest.mark.parametrize("m", [5, 9])
def test_one_cutoff_over(d, m):
    n = 6007
    pts = W.random_blobs(n, d, 90 + d, dup_frac=0.01)
    d0 = 0.01 * d if d <= 4 else 0.04 * d
    cuts = [d0 * (1.0 + 1e-12 * j) for j in range(m)]
    t = torch.from_numpy(pts).cuda()
    got = dpc.dpc_density(t, dpc.Batch.single(n, d, cuts), precision="fp64", sync=True).cpu().numpy()
    assert dpc.dpc_get_stats()["density_layout"] == (5 if d > 1 else 2)
    for c, dc in enumerate(cuts):
        assert np.array_equal(got[c], oracle.density(pts, dc)), c
    check([pts], [[d0] + [d0 * (1.1 + 0.1 * j) for j in range(5)]], "fp64")


def test_instances_disagree_about_the_order():
    insts = [W.random_blobs(n, 3, 95 + n) for n in (5003, 40, 4100, 1)]
    cuts = [[0.02, 0.021, 0.022, 0.023, 0.024], [0.5, 0.1, 0.4, 0.3, 0.01], [0.05, 0.01, 0.2, 0.3, 0.025],
            [1.0, 0.0, 2.0, 3.0, 0.5]]
    check(insts, cuts, "fp64")

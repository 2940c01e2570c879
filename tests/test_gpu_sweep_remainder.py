"""Binary64 densities in segments and pair by pair: both sides of the rule between
them, and sweeps whose levels hold four cutoffs and one over (counted as a
cutoff alone on the group's cells).  Single instances, and a batch whose
instances disagree about which cutoff is the largest.  Exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_2305_11335_gb300 as dpc
import workloads as W
from test_gpu_sweep import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,m,layout", [(6007, d, m, 2) for d in (1, 2, 3, 4, 6) for m in (5, 9)] +
                         [(25568, 2, 5, 2), (25569, 2, 5, 5), (25569, 3, 5, 5), (25569, 6, 5, 5), (25569, 1, 5, 2)])
def test_one_cutoff_over(n, d, m, layout):
    """Segments up to 799 chunks and in 1-D, pairs from 800 on."""
    pts = W.random_blobs(n, d, 90 + d, dup_frac=0.01)
    d0 = (0.01 * d if d <= 4 else 0.04 * d) * (6007 / n) ** (1 / d)
    cuts = [d0 * (1.0 + 1e-12 * j) for j in range(m)]
    t = torch.from_numpy(pts).cuda()
    got = dpc.dpc_density(t, dpc.Batch.single(n, d, cuts), precision="fp64", sync=True).cpu().numpy()
    assert dpc.dpc_get_stats()["density_layout"] == layout
    for c, dc in enumerate(cuts):
        assert np.array_equal(got[c], oracle.density(pts, dc)), c
    if m == 5:
        check([pts], [[d0] + [d0 * (1.1 + 0.2 * j) for j in range(5)]], "fp64")


@pytest.mark.parametrize("n,layout", [(25568, 2), (25569, 5)])
@pytest.mark.parametrize("d", [2, 5])
def test_one_cutoff_on_both_sides_of_the_rule(n, layout, d):
    pts = W.random_blobs(n, d, 99, dup_frac=0.01)
    dc = 0.01 * d
    for ask in ("auto", "segment"):
        got = dpc.dpc_density(torch.from_numpy(pts).cuda(), dpc.Batch.single(n, d, [dc]), precision="fp64", sync=True,
                              layout=ask)
        if ask == "auto":
            assert dpc.dpc_get_stats()["density_layout"] == layout
        assert np.array_equal(got[0].cpu().numpy(), oracle.density(pts, dc))


def test_instances_disagree_about_the_order():
    insts = [W.random_blobs(n, 3, 95 + n) for n in (5003, 40, 4100, 1)]
    cuts = [[0.02, 0.021, 0.022, 0.023, 0.024], [0.5, 0.1, 0.4, 0.3, 0.01], [0.05, 0.01, 0.2, 0.3, 0.025],
            [1.0, 0.0, 2.0, 3.0, 0.5]]
    check(insts, cuts, "fp64")

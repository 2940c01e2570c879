"""Points so close that squared distances are subnormal or vanish in float32
(1e-19 to 1e-25 apart), in binary64 mode and with the float32 filter, against
the oracle: pruning by float32 bounds must leave room for their absolute
error.  Exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_2305_11335_gb300 as dpc
from _gpu_util import assert_same, parity

pytestmark = pytest.mark.gpu


def points(n, d, scale):
    return (np.random.default_rng(d).random((n, d)) * scale).astype(np.float32)


@pytest.mark.parametrize("d", [2, 3, 5])
@pytest.mark.parametrize("scale", [1e-17, 1e-20, 1e-22])
def test_dependent_points_of_close_points(d, scale):
    pts = points(9001, d, scale)
    r = {2: 0.02, 3: 0.06, 5: 0.2}[d] * scale
    parity(pts, [r], rho_noise=2, rho_min=4, delta_min=3.0 * r)
    parity(pts, [r, 1.2 * r], rho_noise=2, rho_min=4, delta_min=3.0 * r)


@pytest.mark.parametrize("layout", ["union", "segment", "tree", "cell"])
def test_near_layouts(layout):
    """Blocks of thousands of points: the passes over the other cells are
    pruned by the best of the own cell."""
    for scale in (1e-20, 1e-22):
        pts = points(9001, 2, scale)
        r = 0.3 * scale
        batch = dpc.Batch.single(9001, 2, [r])
        out = dpc.dpc_run(torch.from_numpy(pts).cuda(), batch, dpc.make_params(batch, 2, 4, r), precision="fp64",
                          layout=layout, sync=True)
        assert_same({k: v[0].cpu().numpy() for k, v in out.items()}, oracle.run(pts, r, 2, 4, r), layout)

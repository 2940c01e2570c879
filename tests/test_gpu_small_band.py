"""Small integer sets whose cutoff many pairs meet exactly (every CTA recounts
its band pairs), and repeated distances for the ranking, against the oracle.
Exact."""
import numpy as np
import pytest

from _gpu_util import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("n", [129, 2500, 8192])
def test_cutoff_met_exactly(n, d):
    extent = {1: 700, 2: 60, 3: 18, 5: 7, 8: 4}[d]
    pts = np.random.default_rng(n + d).integers(-extent, extent, (n, d)).astype(np.int32)
    parity(pts, [5.0, np.sqrt(2.0), 3.0], rho_noise=2, rho_min=5, delta_min=2.0)

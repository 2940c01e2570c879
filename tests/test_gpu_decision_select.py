"""Top-k selection of the decision graph at the edges of its candidate buffer
(4096 points per instance up to 256 instances, by their mean size beyond):
instance sizes around the buffer, masses of equal gamma that overflow it (the exact radix
select), gammas outside the float32 range, and more than 256 instances.
Bit for bit against the oracle (no tolerance)."""
import math

import numpy as np
import pytest

from test_gpu_decision import check, synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4095, 4096, 4097, 20011])
@pytest.mark.parametrize("ties", [False, True])
def test_sizes_around_the_candidate_buffer(n, ties):
    check([n], [synthetic(n, n, ties=ties)], 1000, 24, 48, 0.5)


def test_more_equal_gammas_than_the_buffer_holds():
    n = 30000
    rng = np.random.default_rng(3)
    some = (np.where(rng.random(n) < 0.6, 6, 5).astype(np.int32), np.full(n, 0.5))  # 18000 points at the top value
    some[1][17] = math.inf
    close = (np.full(n, 1000, np.int32), 1.0 + rng.integers(0, 9, n) * 2.0 ** -50)  # equal float32 bounds
    check([n, n, 50], [some, close, synthetic(50, 9)], 700, 8, 16, 0.25)


@pytest.mark.parametrize("scale", [1e-300, 1e-35, 1e38, 1e300])
def test_gammas_outside_float32(scale):
    n = 9000
    rng = np.random.default_rng(4)
    rho = rng.integers(-3, 1 << 20, n).astype(np.int32)
    delta = rng.random(n) * scale
    delta[::97] = 5e-324
    delta[::101] *= -1.0
    check([n], [(rho, delta)], 300, 20, 2048, scale * 1e-3)
    check([n], [(np.abs(rho) + 1, np.abs(delta))], 300, 20, 100, 5e-324)


def test_many_instances():
    sizes = [0, 1] + [40 + 7 * (i % 50) for i in range(300)]
    check(sizes, [synthetic(n, 900 + i, ties=i % 2 == 0) for i, n in enumerate(sizes)], 24, 6, 9, 0.02)


@pytest.mark.parametrize("k", [3, 200, 1000])
@pytest.mark.parametrize("n", [9, 511, 512, 1500, 4095, 4200])
def test_many_instances_of_every_mean_size(n, k):
    sizes = [n + (i * 7) % 5 - 2 for i in range(260)]
    check(sizes, [synthetic(m, 50 + i, ties=i % 3 == 0) for i, m in enumerate(sizes)], k, 6, 9, 0.02)

"""Labels by one CTA per instance or by launches over all points, on both
sides of the rule between them: sizes of one large instance, a few large ones,
counts of tiny instances (with one larger among them), and whole runs of tiny
instances.  Random forests against a sequential walk, cycles reported, the
route read from the launch count."""
import numpy as np
import pytest
import torch

import oracle
import paper_2305_11335_gb300 as dpc
from _gpu_util import assert_same

pytestmark = pytest.mark.gpu

CASES = {  # sizes of the instances, one CTA per instance?
    "one_20480": ([20480], True),
    "one_20481": ([20481], False),
    "one_32768": ([32768], False),
    "sixteen_24000": ([24000] * 16, True),
    "fifteen_24000": ([24000] * 15, False),
    "over_32768": ([32769] + [30000] * 20, False),
    "tiny_4096": ([3] * 4096, True),
    "tiny_4097": ([3] * 4097, False),
    "tiny_and_larger": ([5] * 6000 + [9000, 1], False),
    "many_of_1024": ([1024] * 4100, True),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_forests(name):
    sizes, by_instance = CASES[name]
    rng = np.random.default_rng(len(sizes))
    lam, want = [], []
    for n in sizes:
        i = np.arange(n)
        up = np.maximum(0, i - rng.integers(1, 4, n))  # a chain thousands of links deep
        up[rng.random(n) < 0.002] = -1
        up[0] = -1
        root = i.copy()
        for j in range(n):
            root[j] = j if up[j] < 0 else root[up[j]]
        lam.append(up)
        want.append(root)
    lam, want = np.concatenate(lam).astype(np.int32), np.concatenate(want)
    total = len(lam)
    batch = dpc.Batch.packed(sizes, [2] * len(sizes), [[1.0]] * len(sizes))
    params = dpc.make_params(batch, 0, 1, 1e9)
    rho = torch.ones(total, dtype=torch.int32).cuda()
    delta = torch.zeros(total, dtype=torch.float64).cuda()
    got = dpc.dpc_cluster(batch, 0, params, rho, torch.from_numpy(lam).cuda(), delta, sync=True).cpu().numpy()
    assert np.array_equal(got, want)
    assert (dpc.dpc_get_stats()["kernel_launches"] == 1) == by_instance
    at = int(np.flatnonzero(np.array(sizes) > 1)[-1])  # a cycle of two points in the last instance that can hold one
    o = int(np.sum(sizes[:at]))
    lam[o], lam[o + 1] = 1, 0
    with pytest.raises(dpc.DpcError) as e:
        dpc.dpc_cluster(batch, 0, params, rho, torch.from_numpy(lam).cuda(), delta, sync=True)
    assert e.value.code == dpc.DPC_ERR_DATA


@pytest.mark.parametrize("count,pairs,sweep_pairs,density_pairs", [
    (2048, True, True, True), (4096, True, False, True), (4097, False, False, True), (16385, False, False, False)])
def test_runs_of_tiny_instances(count, pairs, sweep_pairs, density_pairs):
    """Many instances of 20 points on both sides of the all-pairs limits (a run
    by 32-point chunks, a density alone by four times as many)."""
    sizes = [20] * count
    pts = np.random.default_rng(1).random((20 * count, 2), dtype=np.float32)
    batch = dpc.Batch.packed(sizes, [2] * count, [[0.2]] * count)
    t = torch.from_numpy(pts).cuda()
    out = dpc.dpc_run(t, batch, dpc.make_params(batch, 2, 3, 0.3), sync=True)
    assert (dpc.dpc_get_stats()["density_layout"] == 0) == pairs
    out = {k: v[0].cpu().numpy() for k, v in out.items()}
    den = dpc.dpc_density(t, batch, sync=True)[0].cpu().numpy()
    assert (dpc.dpc_get_stats()["density_layout"] == 0) == density_pairs
    assert np.array_equal(den, out["rho"])
    three = dpc.Batch.packed(sizes, [2] * count, [[0.2, 0.3, 0.25]] * count)
    sweep = dpc.dpc_run(t, three, dpc.make_params(three, 2, 3, 0.3), sync=True)
    assert (dpc.dpc_get_stats()["density_layout"] == 0) == sweep_pairs
    sweep = {k: v.cpu().numpy() for k, v in sweep.items()}
    assert_same({k: v[0] for k, v in sweep.items()}, out)
    for i in list(range(0, count, 97)) + [count - 1]:
        s = slice(20 * i, 20 * i + 20)
        assert_same({k: v[s] for k, v in out.items()}, oracle.run(pts[s], 0.2, 2, 3, 0.3), str(i))
        assert_same({k: v[1, s] for k, v in sweep.items()}, oracle.run(pts[s], 0.3, 2, 3, 0.3), str(i))

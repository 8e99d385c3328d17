"""Learning in cells of more than 1 024 records, which one block orders by
radix passes: record counts around a tile of 8 192, one digit and several of
sample ids, sample ids that span more than 24 bits (marked gpu). Eq. 1 in
sample order against plain float64; an order other than the samples' differs
by percents."""
import numpy as np
import pytest

from paper_1911_10217_gb300 import scenes

from .gpu_common import device_scene, params_for
from .test_gpu_descent import env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts,length,skew", [
    ((1025,), 1025, 1.0), ((8191, 5), 8196, 1.0), ((8192,), 8192, 4.0), ((8193, 8192, 1024), 100000, 1.0),
    ((20000, 3000), 23000, 6.0), ((1100, 9000), (1 << 24) + 5000, 1.0),
])
def test_eq1_in_large_cells(env, counts, length, skew):  # noqa: F811
    import torch
    rll, ctx, dev = env["rll"], env["ctx"], env["dev"]
    ctx.sync_status()
    s = scenes.tiny_scene()
    d = device_scene(s, dev)
    alpha = 0.25
    tree = rll.Tree(ctx, d["tri"], d["em"])
    grid = rll.Grid(ctx, tree, params_for(rll, s, alpha=alpha))
    M, m = grid.M, grid.m
    rng = np.random.default_rng(sum(counts))
    at = np.sort(rng.choice(length, sum(counts), replace=False))
    cell = rng.permutation(np.repeat(np.arange(len(counts)), counts))
    cluster = np.minimum((m * rng.uniform(size=at.size) ** skew).astype(np.int64), m - 1)
    val = rng.uniform(0.1, 2.0, at.size).astype(np.float32)
    key = torch.full((length,), -1, dtype=torch.int32, device=dev)
    reward = torch.zeros(length, device=dev)
    idx = torch.from_numpy(at).to(dev)
    key[idx] = torch.from_numpy((cell * M + cluster).astype(np.int32)).to(dev)
    reward[idx] = torch.from_numpy(val).to(dev)
    q0 = grid.export()["q"]
    rll.learn_update(ctx, grid, key, reward)
    assert ctx.sync_status() == 0 and grid.touched_cells() == len(counts)
    q = grid.export()["q"]
    want = q0.astype(np.float64)
    for c, k, v in zip(cell, cluster, val.astype(np.float64)):
        want[c, k] = (1.0 - alpha) * want[c, k] + alpha * v
    # a composed value carries at most some 40 roundings (2^-24 each) of the last records' weight
    assert np.allclose(q[: len(counts), :m], want[: len(counts), :m], rtol=1e-5, atol=0.0)
    assert np.array_equal(q[len(counts):], q0[len(counts):])


@pytest.mark.parametrize("records", [1, 31, 8191, 8193, 16384, 16385])
def test_bucketing_sizes(env, records):  # noqa: F811
    """Up to 16 384 records are bucketed by one cluster of blocks, more by three launches: record
    counts around a round of the cluster (8 192) and its last, twice in a row from the same grid."""
    import torch
    rll, ctx, dev = env["rll"], env["ctx"], env["dev"]
    ctx.sync_status()
    s = scenes.tiny_scene()
    d = device_scene(s, dev)
    alpha = 0.25
    tree = rll.Tree(ctx, d["tri"], d["em"])
    grid = rll.Grid(ctx, tree, params_for(rll, s, alpha=alpha))
    M, m = grid.M, grid.m
    rng = np.random.default_rng(records)
    want = grid.export()["q"].astype(np.float64)
    for turn in range(2):
        key = rng.integers(0, 300, records) * M + rng.integers(0, m, records)
        bad = rng.uniform(size=records) < 0.05
        val = rng.uniform(0.1, 2.0, records).astype(np.float32)
        rll.learn_update(ctx, grid, torch.from_numpy(np.where(bad, -1, key).astype(np.int32)).to(dev),
                         torch.from_numpy(val).to(dev))
        for k, v in zip(key[~bad], val[~bad].astype(np.float64)):
            want[k // M, k % M] = (1.0 - alpha) * want[k // M, k % M] + alpha * v
        assert ctx.sync_status() == 0 and grid.touched_cells() == np.unique(key[~bad] // M).size
        q = grid.export()["q"]
        # some 40 roundings of 2^-24 a turn, see above
        assert np.allclose(q[:, :m], want[:, :m], rtol=2e-5, atol=0.0)

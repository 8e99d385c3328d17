"""Learning calls one after another on the same grid whose large cells come
and go: the kernel of the large cells runs beside the other cells' kernel
where it has cells and hands on at once where it has none, by flags cleared
in every call (marked gpu). Eq. 1 in sample order against plain float64."""
import numpy as np
import pytest

from paper_1911_10217_gb300 import scenes

from .gpu_common import device_scene, params_for
from .test_gpu_descent import env  # noqa: F401

pytestmark = pytest.mark.gpu

# records of a call's largest cell, and of its others (below 16 384 in all one kernel buckets them)
CALLS = [(3000, 500), (0, 700), (9000, 40000), (0, 60000), (0, 700), (2000, 500), (0, 60000), (1025, 60000)]


@pytest.mark.parametrize("turns", [1, 3])
def test_large_cells_come_and_go(env, turns):  # noqa: F811
    import torch
    rll, ctx, dev = env["rll"], env["ctx"], env["dev"]
    ctx.sync_status()
    s = scenes.tiny_scene()
    d = device_scene(s, dev)
    alpha = 0.25
    tree = rll.Tree(ctx, d["tri"], d["em"])
    grid = rll.Grid(ctx, tree, params_for(rll, s, alpha=alpha))
    M, m = grid.M, grid.m
    rng = np.random.default_rng(turns)
    want = grid.export()["q"].astype(np.float64)
    calls = []
    for big, others in CALLS * turns:
        cell = np.concatenate([np.full(big, 7), rng.integers(8, 300, others)])
        cell = cell[rng.permutation(cell.size)]
        cluster = rng.integers(0, m, cell.size)
        val = rng.uniform(0.1, 2.0, cell.size).astype(np.float32)
        calls.append((torch.from_numpy((cell * M + cluster).astype(np.int32)).to(dev), torch.from_numpy(val).to(dev)))
        for c, k, v in zip(cell, cluster, val.astype(np.float64)):
            want[c, k] = (1.0 - alpha) * want[c, k] + alpha * v
    torch.cuda.synchronize()
    for key, val in calls:  # back to back
        rll.learn_update(ctx, grid, key, val)
    assert ctx.sync_status() == 0
    # only the last some 100 records of an entry weigh above the tolerance: as many roundings of 2^-24
    assert np.allclose(grid.export()["q"][:, :m], want[:, :m], rtol=2e-5, atol=0.0)

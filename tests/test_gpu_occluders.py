"""Occluder sets whose table differs from the ordinary one: batches of items
with different box counts (marked gpu)."""
import dataclasses

import numpy as np
import pytest

from paper_1911_10217_gb300 import scenes

from .gpu_common import params_for
from .test_gpu_batched import _build
from .test_gpu_boxes import random_boxes
from .test_gpu_descent import env as _descent_env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(_descent_env):  # noqa: F811
    import torch
    return dict(_descent_env, torch=torch)


@pytest.mark.parametrize("counts", [(257, 256), (200, 320, 1, 256), (0, 1024, 257, 64)])
def test_batch_of_mixed_box_counts(env, counts):
    """A table of 257 boxes is smaller than one of 256 (half the bins): a batch's shared memory holds
    each of its items' tables. The image is the single-grid path's."""
    rll, ctx, torch, dev = env["rll"], env["ctx"], env["torch"], env["dev"]
    sc = []
    for i, n in enumerate(counts):
        s = scenes.frame_scene(seed=60 + i, width=64, height=48, n_patches=8, tris_per_patch=64, n_boxes=32,
                               table_size=1 << 13, cut_size=32, frames=1)
        sc.append(dataclasses.replace(s, boxes=random_boxes(max(n, 1))[:n]))
    objs, batch = _build(env, sc)
    batch.run(do_split=False)
    for o in objs:
        s, d = o["scene"], o["d"]
        g = rll.Grid(ctx, o["tree"], params_for(rll, s))
        n = s.n_points * s.spp
        rgb = torch.empty(3, s.n_points, device=dev)
        key, val = torch.empty(n, dtype=torch.int32, device=dev), torch.empty(n, device=dev)
        rll.sample_and_shade(ctx, g, o["tree"], d["pos"], d["nrm"], d["alb"], d["boxes"], s.seed, 0, s.spp, rgb, key,
                             val)
        # the tolerance of test_batch_matches_single_grid_path
        assert np.allclose(o["rgb"].cpu().numpy(), rgb.cpu().numpy(), rtol=1e-5, atol=1e-9)
    assert ctx.sync_status() == 0

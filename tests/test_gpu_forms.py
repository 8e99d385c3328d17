"""The forms of the sampling kernel that calls without debug outputs take
(one sample a point, a lane a sample, a block's own box table or the call's)
against the oracle (marked gpu). Calls with debug outputs, as in the other
tests, all take one form."""
import dataclasses

import numpy as np
import pytest

from paper_1911_10217_gb300 import scenes

from .gpu_common import compare_samples, device_scene, params_for, run_sample, to_host
from .test_gpu_boxes import random_boxes
from .test_gpu_descent import env  # noqa: F401

pytestmark = pytest.mark.gpu


def scene_of(points, spp, boxes=64):
    s = scenes.frame_scene(seed=11, width=64, height=max(4, -(-points // 64)), n_patches=16, tris_per_patch=64,
                           n_boxes=64, table_size=1 << 15, cut_size=16)
    pick = np.random.default_rng(points).permutation(s.n_points)[:points]
    return dataclasses.replace(s, pos=np.ascontiguousarray(s.pos[:, pick]), nrm=np.ascontiguousarray(s.nrm[:, pick]),
                               albedo=s.albedo[pick], boxes=random_boxes(max(boxes, 1))[:boxes], spp=spp,
                               grid=dataclasses.replace(s.grid, cell_size=0.06))


def check_plain(env, s, option=None, **kw):  # noqa: F811
    """One call without debug outputs into poisoned buffers; light, probabilities and margins from one
    with them on the same state, whose records have to be the same bits."""
    import torch
    O, rll, ctx, dev = env["O"], env["rll"], env["ctx"], env["dev"]
    ctx.sync_status()
    d = device_scene(s, dev)
    ot = O.Tree(s.tris, s.emission)
    dt = rll.Tree(ctx, d["tri"], d["em"])
    og = O.Grid.for_scene(ot, s, **kw)
    dg = rll.Grid(ctx, dt, params_for(rll, s, **kw))
    P, n = s.n_points, s.n_points * s.spp
    rgb = torch.full((3, P), -7.0, device=dev)
    key = torch.full((n,), 0x7ffffff0, dtype=torch.int32, device=dev)
    val = torch.full((n,), -7.0, device=dev)
    try:
        if option:
            ctx.set_option(*option)
        rll.sample_and_shade(ctx, dg, dt, d["pos"], d["nrm"], d["alb"], d["boxes"], s.seed, 3, s.spp, rgb, key, val)
    finally:
        if option:
            ctx.set_option("sample_min_blocks", 4)
    g = to_host(run_sample(rll, ctx, dg, dt, d, s.seed, 3, s.spp))  # every cell is in its slot by now
    plain = to_host(dict(rgb=rgb, key=key, val=val))
    assert np.array_equal(plain["key"], g["key"])
    g.update(plain)
    o = og.sample_frame(O.scene_arrays(s), s.seed, 3, s.spp)
    compare_samples(g, o, dg.export()["keys"], og.keys, dg.M)
    assert ctx.sync_status() == 0


@pytest.mark.parametrize("points,spp", [(1, 2), (37, 3), (33, 31), (5, 32), (7, 33), (2, 65), (1, 1000), (4096, 2),
                                        (8192, 33), (8192, 47), (12000, 65), (20000, 7)])
def test_a_lane_a_sample(env, points, spp):  # noqa: F811
    """Samples a point that do and do not divide a warp; from 8 192 points on a warp takes two points
    and more, so that a round ends one point's sum and begins another's."""
    check_plain(env, scene_of(points, spp))


@pytest.mark.parametrize("points,spp,boxes,mode", [
    (1, 1, 0, "descent"), (5000, 1, 64, "descent"), (5000, 1, 65, "descent"), (160001, 1, 64, "descent"),
    (5000, 1, 64, "descent2"), (5000, 1, 33, "uniform"), (5000, 9, 65, "descent"), (5000, 9, 64, "descent2")])
def test_one_sample_a_point_and_box_tables(env, points, spp, boxes, mode):  # noqa: F811
    """At most 64 boxes and one wave of blocks (155 648 points): each block builds the boxes' table."""
    check_plain(env, scene_of(points, spp, boxes), mode=mode)


@pytest.mark.parametrize("points,spp,mode", [(5000, 9, "descent"), (700, 40, "descent2"), (5000, 1, "descent"),
                                             (90000, 4, "uniform")])
def test_forms_of_the_larger_register_budget(env, points, spp, mode):  # noqa: F811
    """sample_min_blocks = 3 holds for every split of the samples."""
    check_plain(env, scene_of(points, spp), option=("sample_min_blocks", 3), mode=mode)

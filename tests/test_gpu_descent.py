"""The sampling kernel's descent and its work split against the oracle, at the
sizes where they take another path (marked gpu). Light, cell and cluster per
sample exact, continuous values within 1e-4 relative, as in test_gpu_parity."""
import dataclasses

import numpy as np
import pytest

from paper_1911_10217_gb300 import scenes

from .gpu_common import compare_samples, device_scene, params_for, run_sample, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle as O
    from paper_1911_10217_gb300 import rll
    dev = torch.device("cuda:0")
    return dict(O=O, rll=rll, dev=dev, ctx=rll.Context(0, torch.cuda.current_stream(dev)))


def check(env, scene, frames=2, spp=None, builder="lbvh", **kw):
    """Frames of `scene` from the oracle's learned state, sample by sample."""
    O, rll, ctx = env["O"], env["rll"], env["ctx"]
    spp = spp or scene.spp
    ctx.sync_status()
    d = device_scene(scene, env["dev"])
    ot = O.Tree(scene.tris, scene.emission, builder=builder)
    dt = rll.Tree(ctx, d["tri"], d["em"], builder=builder)
    og = O.Grid.for_scene(ot, scene, **kw)
    dg = rll.Grid(ctx, dt, params_for(rll, scene, **kw))
    A = O.scene_arrays(scene)
    for f in range(frames):
        dg.import_state(og.keys, og.cut, og.Q, og.C)
        g = to_host(run_sample(rll, ctx, dg, dt, d, scene.seed, f, spp))
        o = og.sample_frame(A, scene.seed, f, spp)
        compare_samples(g, o, dg.export()["keys"], og.keys, dg.M)
        og.split_collapse(og.learn(o["slot"], o["s"], o["reward"]))
    assert ctx.sync_status() == 0


@pytest.mark.parametrize("mode", ["descent", "descent2"])
@pytest.mark.parametrize("log2_scale", [0, -20])
def test_bounds_at_small_scales(env, mode, log2_scale):
    """At scale 2^-20 the squared distances of the tiny scene lie on both sides
    of 2^-40, below which the bounds take the library's square root."""
    s = scenes.tiny_scene()
    k = np.float32(2.0 ** log2_scale)
    s = dataclasses.replace(s, tris=s.tris * k, boxes=s.boxes * k, pos=s.pos * k,
                            grid=dataclasses.replace(s.grid, cell_size=float(s.grid.cell_size * k)))
    check(env, s, mode=mode)


@pytest.mark.parametrize("points,spp", [(1, 2), (37, 3), (33, 31), (5, 32), (7, 33), (3, 48), (2, 65), (1, 1000),
                                        (4096, 2), (1000, 5)])
def test_samples_split_over_lanes(env, points, spp):
    """More than one sample a point: a lane a sample, points summed across lanes and rounds. Samples a
    point that do and do not divide a warp, points that do not fill one, sums over several rounds."""
    s = scenes.tiny_scene()
    s = dataclasses.replace(s, pos=np.ascontiguousarray(s.pos[:, :points]), nrm=np.ascontiguousarray(s.nrm[:, :points]),
                            albedo=s.albedo[:points])
    check(env, s, spp=spp)

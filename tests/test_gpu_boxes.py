"""The occluder boxes' table (bins and masks) against the oracle, which tests
every box: box counts at the table's steps (64-box words, bins halved above
256), boxes of all sizes, flat ones, one that stretches the bins over a far
larger extent (marked gpu)."""
import dataclasses

import numpy as np
import pytest

from paper_1911_10217_gb300 import scenes

from .test_gpu_descent import check, env  # noqa: F401

pytestmark = pytest.mark.gpu


def random_boxes(n, far=False):
    rng = np.random.default_rng(n)
    size = np.exp(rng.uniform(np.log(2e-3), np.log(0.15), (n, 3)))
    lo = rng.uniform(-0.1, 1.0, (n, 3))
    hi = lo + size
    hi[:: 7, 1] = lo[:: 7, 1]  # flat: never blocks
    if far:
        lo[0], hi[0] = (-1e4, 2.0, -1e4), (1e4, 3.0, 1e4)
    return np.concatenate([lo, hi], axis=1).astype(np.float32)


@pytest.mark.parametrize("n,far", [(1, False), (2, False), (63, False), (64, True), (65, False), (256, False),
                                   (257, True), (1024, False)])
def test_shadow_test_over_the_table(env, n, far):  # noqa: F811
    s = dataclasses.replace(scenes.tiny_scene(), boxes=random_boxes(n, far))
    check(env, s, frames=1, spp=2)


@pytest.mark.parametrize("n,far", [(1, False), (64, True), (257, False), (1024, False)])
def test_bounce_over_the_table(env, n, far):  # noqa: F811
    """Vertices bit for bit, from points inside the room and outside it (paths that escape)."""
    import torch
    O, rll, ctx, dev = env["O"], env["rll"], env["ctx"], env["dev"]
    boxes = random_boxes(n, far)
    rng = np.random.default_rng(5)
    P = 3001
    pos = rng.uniform(-0.3, 1.3, (3, P)).astype(np.float32)
    nrm = rng.normal(size=(3, P))
    nrm[:, :64] = np.eye(3)[:, rng.integers(0, 3, 64)]
    nrm = (nrm / np.linalg.norm(nrm, axis=0)).astype(np.float32)
    oy, on, of = O.bounce_vertices(pos, nrm, boxes, scenes.ROOM, 9, 2, 50.0)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    y, ny, f = torch.empty(3, P, device=dev), torch.empty(3, P, device=dev), torch.empty(P, device=dev)
    rll.bounce_vertices(ctx, t(pos), t(nrm), t(boxes), scenes.ROOM, 9, 2, 50.0, y, ny, f)
    for got, want in ((y, oy), (ny, on), (f, of)):
        assert np.array_equal(got.cpu().numpy(), np.asarray(want, np.float32))


@pytest.mark.parametrize("lights,boxes", [(1, 64), (2, 64), (3, 0), (400, 65), (512, 64), (513, 256), (4096, 1024)])
def test_energy_sampler_search(env, lights, boxes):  # noqa: F811
    """The light search's first nine probes come from shared memory: fewer lights than they tell
    apart, as many, and more. The chosen light is the first whose prefix exceeds the draw."""
    import torch
    O, rll, ctx, dev = env["O"], env["rll"], env["ctx"], env["dev"]
    s = scenes.frame_scene(seed=3, width=64, height=32, n_patches=16, tris_per_patch=256, n_boxes=32)
    tris, emission = s.tris[:lights], s.emission[:lights]
    s = dataclasses.replace(s, tris=tris, emission=emission, boxes=random_boxes(boxes))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    tree = rll.Tree(ctx, t(tris.reshape(-1, 9)), t(emission))
    ot = O.Tree(tris, emission)
    P, spp = s.n_points, 5
    rgb, light = torch.empty(3, P, device=dev), torch.empty(P * spp, dtype=torch.int32, device=dev)
    rll.sample_power(ctx, tree, t(s.pos), t(s.nrm), t(s.albedo), t(s.boxes), 3, 0, spp, rgb, light)
    orgb, olight = O.sample_power(ot, O.scene_arrays(s), 3, 0, spp)
    lg = light.cpu().numpy()
    # the device's prefix sums are binary32: draws within their rounding of a boundary may differ
    assert np.mean(lg != olight) < 1e-3 and np.abs(lg - olight).max() <= 1
    same = np.all((lg == olight).reshape(P, spp), axis=1)
    assert np.allclose(rgb.cpu().numpy()[:, same], orgb[:, same], rtol=1e-3, atol=1e-7)


@pytest.mark.parametrize("n_boxes", [0, 64, 1024])
def test_blocks_that_take_many_points(env, n_boxes):  # noqa: F811
    """Energy sampler and bounces of more points than fit the device at once, in blocks that stride over
    them: any point's result is the one it has in a call of few points, bit for bit."""
    import torch
    rll, ctx, dev = env["rll"], env["ctx"], env["dev"]
    s = scenes.tiny_scene()
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    tree = rll.Tree(ctx, t(s.tris.reshape(-1, 9)), t(s.emission))
    boxes = t(random_boxes(max(n_boxes, 1))[:n_boxes])
    rng = np.random.default_rng(8)
    P, few = 1_000_003, 5001  # 152 SMs hold at most 311 296 threads
    pos = rng.uniform(0.0, 1.0, (3, P)).astype(np.float32)
    nrm = rng.normal(size=(3, P))
    nrm = (nrm / np.linalg.norm(nrm, axis=0)).astype(np.float32)
    alb = rng.uniform(0.1, 0.9, P).astype(np.float32)

    def run(p):
        x, n = t(pos[:, :p]), t(nrm[:, :p])
        out = [torch.full((3, p), -7.0, device=dev) for _ in range(3)] + [torch.full((p,), -7.0, device=dev)]
        rll.sample_power(ctx, tree, x, n, t(alb[:p]), boxes, 3, 1, 2, out[0])
        rll.bounce_vertices(ctx, x, n, boxes, scenes.ROOM, 9, 2, 50.0, out[1], out[2], out[3])
        return [a.cpu().numpy() for a in out]

    large, small = run(P), run(few)
    for a, b in zip(large, small):
        assert np.array_equal(a[..., :few], b)
    # the others: outputs depend on the point's index through the draws alone; all are written
    assert all(not np.any(a == -7.0) for a in large)

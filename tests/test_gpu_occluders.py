"""Occluder sets that the ordinary ones leave out: batches of items
with different box counts, boxes met at the same distance, boxes
given with minimum and maximum exchanged, few boxes, boxes that reach far out
of the room (marked gpu)."""
import dataclasses

import numpy as np
import pytest

from paper_1911_10217_gb300 import scenes

from .gpu_common import device_scene, params_for
from .test_gpu_batched import _build
from .test_gpu_boxes import random_boxes
from .test_gpu_descent import check, env as _descent_env  # noqa: F401

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


def bounce_ray(O, x, n, seed, point, frame):
    """Origin, direction and reciprocal of a point's bounce in binary32, for a normal (0, 1, 0): the
    tangent frame is (0, 0, -1), (-1, 0, 0)."""
    f = np.float32
    a = b = f(0)
    for k in range(16):
        w = O.philox4x32_10([point, frame, k >> 1, 1], [seed, 0])
        ta, tb = (f(2) * (f(int(w[2 * (k & 1) + j]) >> 8) * f(2.0 ** -24)) - f(1) for j in (0, 1))
        if f(ta * ta) + f(tb * tb) < f(1):
            a, b = ta, tb
            break
    c = np.sqrt(f(1) - f(f(a * a) + f(b * b)))
    d = np.array([-b, c, -a], f)
    return np.asarray(x, f) + f(1e-4) * np.asarray(n, f), d, f(1) / d


def test_bounce_on_two_boxes_at_the_same_distance(env):
    """A ray that meets a side of one box and the underside of another at the same binary32 distance,
    beyond the first segment: the box of the lower index counts, also where the other one reaches back
    to the ray's origin and is tested first."""
    O, rll, ctx, torch, dev = env["O"], env["rll"], env["ctx"], env["torch"], env["dev"]
    f = np.float32
    x, n, seed, frame, P = [0.51, 0.05, 0.5], [0.0, 1.0, 0.0], 9, 2, 4000
    pos, nrm = (np.repeat(np.array(v, f)[:, None], P, 1) for v in (x, n))
    corners = np.tile(np.array([[0, 0, 0, .01, .01, .01], [.99, .99, .99, 1, 1, 1]], f), (20, 1))  # many boxes
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    tried = 0
    for p in range(P):
        o, d, inv = bounce_ray(O, x, n, seed, p, frame)
        if not (0.01 < d[0] < 0.02 and abs(d[2]) < 0.5 and tried < 4):
            continue
        for y in np.linspace(0.6, 0.7, 400, dtype=f):
            T = f(y - o[1]) * inv[1]
            side = f(o[0] + T * d[0]) + np.arange(-40, 41).astype(f) * f(2.0 ** -24)
            side = side[(side - o[0]).astype(f) * inv[0] == T]
            if side.size:
                break
        else:
            continue
        tried += 1
        z = float(o[2] + T * d[2])
        above = np.array([o[0] - 0.02, y, z - 0.02, o[0] + 0.05, y + 0.1, z + 0.02], f)  # far from the origin
        beside = np.array([side[0], 0.0, 0.0, side[0] + f(0.3), 1.0, 1.0], f)             # along the ray
        axes = []
        for boxes in ([above, beside, *corners], [*corners, beside, above]):
            boxes = np.array(boxes, f)
            want = [np.asarray(a, f) for a in O.bounce_vertices(pos, nrm, boxes, scenes.ROOM, seed, frame, 50.0)]
            out = [torch.empty(3, P, device=dev), torch.empty(3, P, device=dev), torch.empty(P, device=dev)]
            rll.bounce_vertices(ctx, t(pos), t(nrm), t(boxes), scenes.ROOM, seed, frame, 50.0, *out)
            for got, w in zip(out, want):
                assert np.array_equal(got.cpu().numpy(), w)
            axes.append(int(np.argmax(np.abs(want[1][:, p]))))
        assert axes == [1, 0]  # the two are at the same distance indeed
    assert tried >= 2


def swapped(boxes, seed):
    """Every other box with minimum and maximum exchanged along some axes."""
    rng = np.random.default_rng(seed)
    out = boxes.copy()
    for b in range(0, len(out), 2):
        for k in range(3):
            if rng.uniform() < 0.5:
                out[b, k], out[b, 3 + k] = boxes[b, 3 + k], boxes[b, k]
    return out


@pytest.mark.parametrize("n", [1, 64, 300])
def test_bounce_on_boxes_the_other_way_round(env, n):
    """The slab test takes a box with minimum and maximum exchanged like any other."""
    O, rll, ctx, torch, dev = env["O"], env["rll"], env["ctx"], env["torch"], env["dev"]
    boxes = swapped(random_boxes(n), n)
    rng = np.random.default_rng(4)
    P = 4001
    pos = rng.uniform(0.0, 1.0, (3, P)).astype(np.float32)
    nrm = rng.normal(size=(3, P))
    nrm = (nrm / np.linalg.norm(nrm, axis=0)).astype(np.float32)
    want = O.bounce_vertices(pos, nrm, boxes, scenes.ROOM, 9, 2, 50.0)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    out = [torch.empty(3, P, device=dev), torch.empty(3, P, device=dev), torch.empty(P, device=dev)]
    rll.bounce_vertices(ctx, t(pos), t(nrm), t(boxes), scenes.ROOM, 9, 2, 50.0, *out)
    for got, w in zip(out, want):
        assert np.array_equal(got.cpu().numpy(), np.asarray(w, np.float32))


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_shadow_of_a_box_the_other_way_round(env, axis):
    """To the shadow test a box with minimum and maximum exchanged along an axis counts where the segment
    spans all of it: one from far beyond the room to far before it never does."""
    rll, ctx, torch, dev = env["rll"], env["ctx"], env["torch"], env["dev"]
    s = scenes.small_frame_scene()
    d = device_scene(s, dev)
    tree = rll.Tree(ctx, d["tri"], d["em"])
    one = np.array([[.45, .45, .45, .55, .55, .55]], np.float32)  # the bins are cut over this one
    far = np.array([[-10, -10, -10, 10, 10, 10]], np.float32)
    far[0, [axis, 3 + axis]] = 10, -10
    images = []
    for boxes in (one, np.concatenate([one, far])):
        b = torch.from_numpy(boxes).to(dev)
        grid = rll.Grid(ctx, tree, params_for(rll, s))
        rgb, power = torch.empty(3, s.n_points, device=dev), torch.empty(3, s.n_points, device=dev)
        rll.sample_and_shade(ctx, grid, tree, d["pos"], d["nrm"], d["alb"], b, 5, 0, 1, rgb)
        rll.sample_power(ctx, tree, d["pos"], d["nrm"], d["alb"], b, 5, 0, 1, power)
        images.append((rgb.cpu().numpy(), power.cpu().numpy()))
    for a, b in zip(*images):
        assert np.count_nonzero(a) > 100 and np.array_equal(a, b)


def test_shadow_of_a_spanned_box(env):
    """A thin wall given the other way round blocks the segments that cross all of it, like the wall
    itself; only segments that end inside it (a thousandth of the room) may differ."""
    rll, ctx, torch, dev = env["rll"], env["ctx"], env["torch"], env["dev"]
    s = scenes.small_frame_scene()
    d = device_scene(s, dev)
    tree = rll.Tree(ctx, d["tri"], d["em"])
    wall = np.array([[.4995, -1, -1, .5005, 2, 2]], np.float32)
    images = []
    for boxes in (wall[:0], wall, wall[:, [3, 1, 2, 0, 4, 5]]):
        b = torch.from_numpy(np.ascontiguousarray(boxes)).to(dev)
        rgb = torch.empty(3, s.n_points, device=dev)
        rll.sample_power(ctx, tree, d["pos"], d["nrm"], d["alb"], b, 5, 0, 1, rgb)
        images.append(rgb.cpu().numpy())
    blocked = np.any(images[0] != images[1], axis=0)
    assert np.mean(blocked) > 0.2
    assert np.mean(np.all(images[1] == images[2], axis=0)) > 0.99


@pytest.mark.parametrize("points,n", [(300, 0), (300, 20), (300, 21), (300, 32), (300, 33), (45000, 0), (45000, 1),
                                      (45000, 20), (45000, 21)])
def test_bounce_over_few_boxes(env, points, n):
    """Up to 20 boxes, or 32 in launches of at most a block an SM (38 912 points), are tested in turn;
    more over the table."""
    O, rll, ctx, torch, dev = env["O"], env["rll"], env["ctx"], env["torch"], env["dev"]
    boxes = random_boxes(max(n, 1))[:n]
    rng = np.random.default_rng(n)
    pos = rng.uniform(-0.1, 1.1, (3, points)).astype(np.float32)
    nrm = rng.normal(size=(3, points))
    nrm = (nrm / np.linalg.norm(nrm, axis=0)).astype(np.float32)
    want = O.bounce_vertices(pos, nrm, boxes, scenes.ROOM, 9, 2, 50.0)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    out = [torch.empty(3, points, device=dev), torch.empty(3, points, device=dev), torch.empty(points, device=dev)]
    rll.bounce_vertices(ctx, t(pos), t(nrm), t(boxes), scenes.ROOM, 9, 2, 50.0, *out)
    for got, w in zip(out, want):
        assert np.array_equal(got.cpu().numpy(), np.asarray(w, np.float32))


def stretched_boxes(kind, n):
    """n boxes of which a few lie or reach far out of the room."""
    b = random_boxes(n)
    far = np.float32(3e38 if kind == "huge" else np.inf)
    if kind == "slab":
        b[-1] = (-100, -1.1, -100, 100, -1, 100)
    elif kind == "walls":
        b[-4:] = [(-9, -9, -9, 9, -8.9, 9), (-9, 8.9, -9, 9, 9, 9), (-9, -9, -9, -8.9, 9, 9), (8.9, -9, -9, 9, 9, 9)]
    elif kind in ("huge", "endless"):
        b[-1], b[0] = (-far, .9, -far, far, far, far), (-far, -far, -far, -.2, far, far)
    elif kind == "steps":  # ever farther
        for i in range(min(n // 4, 20)):
            b[i] += np.float32(4.0 ** i)
    elif kind == "alike":  # ends that no bins tell apart, but for two
        b[2:] = (.4, .4, .4, .4, .6, .6)
    return b


@pytest.mark.parametrize("n", [16, 17, 64, 300])
@pytest.mark.parametrize("kind", ["slab", "walls", "huge", "endless", "steps", "alike"])
def test_bins_that_few_boxes_would_stretch(env, kind, n):
    """The bins are cut over the range of most boxes: samples and vertices against the oracle, which
    tests every box."""
    O, rll, ctx, torch, dev = env["O"], env["rll"], env["ctx"], env["torch"], env["dev"]
    boxes = stretched_boxes(kind, n)
    check(env, dataclasses.replace(scenes.tiny_scene(), boxes=boxes), frames=1, spp=2)
    rng = np.random.default_rng(7)
    P = 3001
    pos = rng.uniform(-0.3, 1.3, (3, P)).astype(np.float32)
    nrm = rng.normal(size=(3, P))
    nrm[:, :64] = np.eye(3)[:, rng.integers(0, 3, 64)]
    nrm = (nrm / np.linalg.norm(nrm, axis=0)).astype(np.float32)
    want = O.bounce_vertices(pos, nrm, boxes, scenes.ROOM, 9, 2, 50.0)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    out = [torch.empty(3, P, device=dev), torch.empty(3, P, device=dev), torch.empty(P, device=dev)]
    rll.bounce_vertices(ctx, t(pos), t(nrm), t(boxes), scenes.ROOM, 9, 2, 50.0, *out)
    for got, w in zip(out, want):
        assert np.array_equal(got.cpu().numpy(), np.asarray(w, np.float32))

"""The work that programs give this library, as measurable cases.

A case is one pass of a kind of program: sample the shading points of a frame
and learn from what the last one saw (`pass`), the same from host buffers
(`host`), with path vertices (`paths`), many scenes at once (`batch`), or the
energy-based baseline sampler (`power`). A learning pass first applies the
last frame's records to the tables and then samples the next frame, so that
its image and records show the tables that it just wrote.

State starts as a learned one: a few passes run, are exported, and are
imported again with the cells in a fixed order. (Two cells that hash to the
same slot take their places in the order of arrival, so slots, and with them
the record keys, differ from run to run otherwise.)

Sampled outputs have no 64-bit counterpart: each follows from binary32
comparisons with random draws (cell, cluster, light, visibility), where a
value a rounding away gives another light. `exact` covers the geometry of the
path vertices.
"""
import math

import numpy as np
import torch

from paper_1911_10217_gb300 import rll, scenes

DEV = "cuda:0"
LEARN_PASSES = 4            # passes behind a prepared state
CELLS_PER_PX2 = 21.0        # cells that jittered lookups touch, per cell-sized square of pixels


def _pass(name, **kw):
    c = dict(name=name, kind="pass", scene="walled", width=1920, height=1080, spp=1, patches=64, patch_tris=1024,
             boxes=64, cut=32, table=1 << 20, cell_px=30, precision="fp32", mode="descent", tree="lbvh", levels=1,
             split="fused", split_iterations=1, blink=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: a thumbnail of a small room, where launches and host work count
        _pass("tiny_64x64", scene="tiny", width=64, height=64, spp=4, patches=4, patch_tris=64, boxes=8, cut=16,
              table=1 << 10, cell_px=8),
        # an interactive preview at an odd size with a small light set
        _pass("preview_641x359", width=641, height=359, patches=16, patch_tris=256, boxes=32, table=1 << 16,
              cell_px=20),
        # the headline: a static 1080p frame, 64K lights, 32-leaf cuts, one sample a point
        _pass("frame_1080p"),
        # dynamic lighting at 4K: a million lights, a tenth blinking, 64-leaf cuts in bfloat16
        _pass("dynamic_4k_bf16", width=3840, height=2160, patches=1024, cut=64, table=1 << 21, precision="bf16",
              blink=True),
        # the same frame by a renderer that keeps its G-buffer and image in page-locked host memory
        _pass("host_1080p", kind="host"),
        # path tracing: primary points and one bounce each, cells sized by footprint over eight levels
        _pass("paths_720p", kind="paths", width=1280, height=720, patches=32, patch_tris=512, table=1 << 17,
              levels=8),
        # an interior lit by a sky dome and a sun through small openings, 128-leaf cuts in binary16
        _pass("sky_1080p_m128_fp16", scene="sky", spp=2, patches=1, patch_tris=2050, boxes=64, cut=128,
              table=1 << 15, cell_px=30, precision="fp16"),
        # a final-quality tile: many samples a point, so that cells hold thousands of records; 256-leaf
        # cuts, learning and iterated split-collapse as two calls
        _pass("tile_200x120_64spp_m256", width=200, height=120, spp=64, patches=64, patch_tris=256, cut=256,
              table=1 << 15, cell_px=20, split="calls", split_iterations=4),
        # two levels a step over a surface-area-orientation tree, binary16 tables, an odd frame
        _pass("descent2_saoh_1601x901", width=1601, height=901, patches=64, patch_tris=512, precision="fp16",
              mode="descent2", tree="saoh", table=1 << 18),
        # many uneven scenes in one recorded pass
        _pass("batch_12_scenes", kind="batch", scenes=12, replay=True, width=512, height=512, patches=32,
              patch_tris=256, boxes=32, table=1 << 16, cell_px=30),
        # a serving step: a few sessions whose frames happen to be due together, set up anew each time
        _pass("serve_3_sessions_bf16", kind="batch", scenes=3, replay=False, width=960, height=540, patches=64,
              patch_tris=256, boxes=64, table=1 << 18, cell_px=30, precision="bf16"),
        # the energy-based baseline that a learned image is compared with
        _pass("power_1080p_4spp", kind="power", spp=4, table=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same kinds: sizes over the range of the listed ones, options mixed."""
    kind = rng.choice(["pass", "pass", "pass", "host", "paths", "batch", "power"])
    points = _log_int(rng, 2000, 4000000 if kind == "pass" else 1500000)
    width = max(16, int(math.sqrt(points * rng.uniform(1.0, 2.4))))
    height = max(16, points // width)
    spp = 1 if points > 1000000 else _log_int(rng, 1, min(48, max(2, 2000000 // points)))
    c = _pass("drawn", kind=kind, width=width, height=height, spp=spp, patches=_log_int(rng, 4, 256),
              patch_tris=2 * _log_int(rng, 8, 512), boxes=rng.randint(24, 160),
              cut=rng.choice([16, 24, 32, 50, 64, 128, 256]), cell_px=rng.randint(16, 48),
              precision=rng.choice(["fp32", "fp32", "bf16", "fp16"]),
              mode=rng.choice(["descent", "descent", "descent", "descent2", "uniform"]),
              tree=rng.choice(["lbvh", "lbvh", "saoh", "median"]), split=rng.choice(["fused", "fused", "calls"]),
              split_iterations=rng.choice([1, 1, 1, 4]), blink=rng.random() < 0.3)
    if kind == "pass" and rng.random() < 0.25:
        c.update(scene="sky", patches=1, patch_tris=2050, boxes=64)
    if kind == "paths":
        c["levels"] = rng.choice([4, 8])
    if kind == "batch":
        c.update(scenes=rng.randint(2, 10), replay=rng.random() < 0.5, cut=rng.choice([16, 32, 64]), spp=1,
                 width=max(16, min(700, width)), height=max(16, min(400, height)))
    if kind == "power":
        c["table"] = 16
    else:
        cells = min(CELLS_PER_PX2 * width * height / c["cell_px"] ** 2, 1.0 * width * height * c["spp"])
        c["table"] = 1 << max(11, min(20, int(math.ceil(math.log2(16.0 * cells)))))  # far from full
        while c["table"] * c["levels"] * c["cut"] > 1 << 26:
            c["table"] //= 2
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _planes(seed, width, height):
    """The walled room's G-buffer (scenes.frame_scene's recipe) made on the GPU: points on 16 tilted
    planes, one a cell, normals within 15 degrees of the plane's, albedo U[0.2, 0.9]."""
    rng = np.random.default_rng(seed + 77)
    g = torch.Generator(device=DEV).manual_seed(seed)
    frames = np.zeros((16, 12))
    for k in range(16):
        ang, phi = math.radians(30.0) * math.sqrt(rng.uniform()), rng.uniform(0.0, 2.0 * math.pi)
        n = np.array([math.sin(ang) * math.cos(phi), math.cos(ang), math.sin(ang) * math.sin(phi)])
        u = np.cross(n, [1.0, 0.0, 0.0])
        u /= np.linalg.norm(u)
        frames[k] = np.concatenate([n, u, np.cross(n, u),
                                    [(k % 4 + 0.5) / 4.0, rng.uniform(0.0, 0.25), (k // 4 + 0.5) / 4.0]])
    x, y = torch.arange(width, device=DEV).repeat(height), torch.arange(height, device=DEV).repeat_interleave(width)
    bw, bh = max(1, width // 4), max(1, height // 4)
    px, py = torch.clamp(x // bw, max=3), torch.clamp(y // bh, max=3)
    f = torch.from_numpy(frames).to(DEV, torch.float32)[px + 4 * py].T      # [12, P]
    su = (x - px * bw + 0.5) / torch.where(px < 3, bw, width - 3 * bw) - 0.5
    sv = (y - py * bh + 0.5) / torch.where(py < 3, bh, height - 3 * bh) - 0.5
    pos = (f[9:12] + 0.175 * (su * f[3:6] + sv * f[6:9])).contiguous()
    z = 1.0 - torch.rand(width * height, device=DEV, generator=g) * (1.0 - math.cos(math.radians(15.0)))
    phi = torch.rand(width * height, device=DEV, generator=g) * (2.0 * math.pi)
    r = torch.sqrt(1.0 - z * z)
    nrm = r * torch.cos(phi) * f[3:6] + r * torch.sin(phi) * f[6:9] + z * f[0:3]
    nrm = (nrm / nrm.norm(dim=0)).contiguous()
    alb = 0.2 + 0.7 * torch.rand(width * height, device=DEV, generator=g)
    return pos, nrm, alb


def _scene(c, seed):
    """Device arrays and grid configuration of one scene."""
    W, H = c["width"], c["height"]
    if c["scene"] == "tiny":
        s = scenes.tiny_scene(seed)
    elif c["scene"] == "sky":
        s = scenes.sky_scene(seed, width=W, height=H, cell_size=c["cell_px"] / W, sun=True)
    else:
        s = scenes.frame_scene(seed, width=16, height=16, n_patches=c["patches"], tris_per_patch=c["patch_tris"],
                               n_boxes=c["boxes"])
        s.grid.cell_size = 0.7 * c["cell_px"] / W
    d = dict(tri=torch.from_numpy(s.tris.reshape(-1, 9)).to(DEV), em=torch.from_numpy(s.emission).to(DEV),
             boxes=torch.from_numpy(s.boxes).to(DEV), boxes_host=s.boxes, grid=s.grid)
    if c["scene"] == "walled":
        d["pos"], d["nrm"], d["alb"] = _planes(seed, W, H)
    else:
        d["pos"], d["nrm"], d["alb"] = (torch.from_numpy(a).to(DEV) for a in (s.pos, s.nrm, s.albedo))
    d["frames_em"] = [d["em"]]
    if c["blink"]:  # radiance of four instants; the tree is built for the largest
        g = torch.Generator(device=DEV).manual_seed(seed + 1)
        n = d["em"].shape[0]
        on = torch.rand(n, device=DEV, generator=g) < 0.1
        ph = torch.rand(n, device=DEV, generator=g) * (2.0 * math.pi)
        d["frames_em"] = [d["em"] * torch.where(on, 1.0 + 0.9 * torch.sin(ph + 1.3 * k), 1.0)[:, None]
                          for k in range(4)]
        d["em"] = d["em"] * torch.where(on, 1.9, 1.0)[:, None]
    return d


def _params(c, d):
    return rll.grid_params_for(d["grid"], table_size=c["table"], cut_size=c["cut"], precision=c["precision"],
                               mode=c["mode"], levels=c["levels"], split_iterations=c["split_iterations"])


def _in_fixed_order(grid, table):
    """Exports the learned state and imports it with every level's cells inserted in increasing order of key."""
    s = grid.export()
    occ = np.nonzero(s["keys"] != np.uint64(0xFFFFFFFFFFFFFFFF))[0]
    occ = occ[np.lexsort((s["keys"][occ], occ // table))]
    with np.errstate(over="ignore"):
        h = s["keys"][occ]
        for mul in (0xFF51AFD7ED558CCD, 0xC4CEB9FE1A85EC53):
            h = (h ^ (h >> np.uint64(33))) * np.uint64(mul)
        h = h ^ (h >> np.uint64(33))
    home = (h & np.uint64(table - 1)).astype(np.int64).tolist()
    slots, taken = [], set()
    for base, at in zip((occ // table * table).tolist(), home):
        while base + at in taken:
            at = (at + 1) & (table - 1)
        taken.add(base + at)
        slots.append(base + at)
    out = dict(keys=np.full_like(s["keys"], 0xFFFFFFFFFFFFFFFF), cut=np.zeros_like(s["cut"]),
               q=np.zeros_like(s["q"]), c=np.zeros_like(s["c"]))
    for k in out:
        out[k][slots] = s[k][occ]
    grid.import_state(out["keys"], out["cut"], out["q"], out["c"])


# ---------------------------------------------------------------- the kinds of program
def _learn(s):
    if s["case"]["split"] == "fused":
        rll.learn_update_split(s["ctx"], s["grid"], s["tree"], s["key"], s["val"])
    else:
        rll.learn_update(s["ctx"], s["grid"], s["key"], s["val"])
        rll.split_collapse(s["ctx"], s["grid"], s["tree"])


def _shade(s):
    """One frame's sampling into the state's buffers."""
    d, f, spp, P = s["d"], s["frame"], s["case"]["spp"], s["d"]["alb"].shape[0]
    s["frame"] = f + 1
    if len(d["frames_em"]) > 1:
        s["tree"].update_emission(d["frames_em"][f % 4])
    if s["case"]["kind"] != "paths":
        rll.sample_and_shade(s["ctx"], s["grid"], s["tree"], d["pos"], d["nrm"], d["alb"], d["boxes"], s["seed"], f,
                             spp, s["rgb"], s["key"], s["val"])
        return [s["rgb"], s["key"], s["val"]]
    n = P * spp
    rll.bounce_vertices(s["ctx"], d["pos"], d["nrm"], d["boxes"], scenes.ROOM, s["seed"], f, 100.0, s["bpos"],
                        s["bnrm"], s["bfp"])
    rll.sample_and_shade(s["ctx"], s["grid"], s["tree"], d["pos"], d["nrm"], d["alb"], d["boxes"], s["seed"], f, spp,
                         s["rgb"], s["key"][:n], s["val"][:n], footprint=s["fp"])
    rll.sample_and_shade(s["ctx"], s["grid"], s["tree"], s["bpos"], s["bnrm"], d["alb"], d["boxes"], s["seed"] + 1, f,
                         spp, s["brgb"], s["key"][n:], s["val"][n:], footprint=s["bfp"])
    return [s["bpos"], s["bnrm"], s["bfp"], s["rgb"], s["brgb"], s["key"], s["val"]]


def _prepare_batch(c, seed):
    ctx = rll.Context(0, torch.cuda.current_stream())
    items, keep = [], []
    for i in range(c["scenes"]):  # uneven: sides from half to twice the case's, and as many lights
        a, b = 2.0 ** (1.0 - 2.0 * (i * 0.618 % 1.0)), 2.0 ** (1.0 - 2.0 * (i * 0.414 % 1.0))
        ci = dict(c, width=max(16, int(c["width"] * a)), height=max(16, int(c["height"] * b)),
                  patches=max(4, int(c["patches"] * a)), cut=c["cut"] if i % 3 else max(16, c["cut"] // 2))
        d = _scene(ci, seed * 131 + i)
        tree = rll.Tree(ctx, d["tri"], d["em"], builder=c["tree"])
        grid = rll.Grid(ctx, tree, _params(ci, d))
        rgb = torch.zeros_like(d["pos"])
        items.append(dict(grid=grid, tree=tree, pos=d["pos"], nrm=d["nrm"], albedo=d["alb"], boxes=d["boxes"],
                          seed=seed + i, frame=0, spp=c["spp"], rgb=rgb))
        keep.append(d)
    batch = rll.Batch(ctx, items)
    for _ in range(LEARN_PASSES):
        batch.run(True)
    if c["replay"]:
        batch.capture(True)
    return dict(case=c, ctx=ctx, batch=batch, items=items, keep=keep, frame=LEARN_PASSES)


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        return _prepare_batch(c, seed)
    ctx = rll.Context(0, torch.cuda.current_stream())
    d = _scene(c, seed)
    tree = rll.Tree(ctx, d["tri"], d["em"], builder=c["tree"])
    P = d["alb"].shape[0]
    s = dict(case=c, ctx=ctx, d=d, tree=tree, seed=seed + 5, frame=0, rgb=torch.zeros(3, P, device=DEV))
    if c["kind"] == "power":
        s["light"] = torch.zeros(P * c["spp"], dtype=torch.int32, device=DEV)
        return s
    s["grid"] = grid = rll.Grid(ctx, tree, _params(c, d))
    n = P * c["spp"] * (2 if c["kind"] == "paths" else 1)
    s["key"], s["val"] = torch.zeros(n, dtype=torch.int32, device=DEV), torch.zeros(n, device=DEV)
    if c["kind"] == "paths":
        s.update(bpos=torch.zeros(3, P, device=DEV), bnrm=torch.zeros(3, P, device=DEV),
                 bfp=torch.zeros(P, device=DEV), brgb=torch.zeros(3, P, device=DEV),
                 fp=torch.full((P,), d["grid"].cell_size, device=DEV))
    for _ in range(LEARN_PASSES):
        _shade(s)
        _learn(s)
    _in_fixed_order(grid, c["table"])
    if c["kind"] == "host":
        s["host"] = [t.cpu().pin_memory() for t in (d["pos"], d["nrm"], d["alb"], s["rgb"])]
    else:
        _shade(s)
    return s


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "batch":
        if c["replay"]:
            s["batch"].launch()
        else:
            for it in s["items"]:
                it["frame"] = s["frame"]
            s["batch"].set_items(s["items"])
            s["batch"].run(True)
        s["frame"] += 1
        return [it["rgb"] for it in s["items"]]
    if c["kind"] == "power":
        d = s["d"]
        rll.sample_power(s["ctx"], s["tree"], d["pos"], d["nrm"], d["alb"], d["boxes"], s["seed"], s["frame"],
                         c["spp"], s["rgb"], s["light"])
        s["frame"] += 1
        return [s["rgb"], s["light"]]
    if c["kind"] == "host":
        pos, nrm, alb, rgb = s["host"]
        rll.render_pass_host(s["ctx"], s["grid"], s["tree"], pos, nrm, alb, s["d"]["boxes_host"], s["seed"],
                             s["frame"], c["spp"], rgb)
        s["frame"] += 1
        return [rgb]
    _learn(s)
    return _shade(s)


def work(case):
    """Bytes: G-buffer and image (40 a point), records written and read again (16 a sample), the rows of
    the touched cells (node ids, Q and C, read and written where learning does). Operations: a sample's
    cell, search, light point and shading (about 250), 90 a descent level (two bounds), and the few boxes
    around its segment."""
    c = case
    P, scale = c["width"] * c["height"], c.get("scenes", 1) * (2 if c["kind"] == "paths" else 1)
    S, lights = P * c["spp"], c["patches"] * c["patch_tris"]
    if c["kind"] == "power":
        return {"bytes": 40.0 * P + 4.0 * S, "flops": S * (150.0 + 2.0 * math.log2(lights) + 72.0)}
    cells = min(CELLS_PER_PX2 * P / c["cell_px"] ** 2, 1.0 * S, 1.0 * c["table"] * c["levels"])
    row = c["cut"] * (20.0 if c["precision"] == "fp32" else 14.0)
    levels = 0.0 if c["mode"] == "uniform" else max(0.0, math.log2(lights / c["cut"]))
    return {"bytes": scale * (40.0 * P + 16.0 * S + cells * row),
            "flops": scale * S * (250.0 + 90.0 * levels + 72.0)}


# ---------------------------------------------------------------- 64-bit values
def _philox_words(idx, frame, block, seed):
    """The four words of Philox4x32-10 for counter (idx, frame, block, 1) and a 64-bit key (Salmon et al., SC'11)."""
    m = 0xFFFFFFFF
    c = [idx.to(torch.int64), torch.full_like(idx, frame), torch.full_like(idx, block), torch.full_like(idx, 1)]
    k = [seed & m, (seed >> 32) & m]

    def mul(a, b):  # high and low words of a 32 x 32-bit product, in halves of 16 bits
        lo, hi = (b & 0xFFFF) * a, (b >> 16) * a
        s = lo + ((hi & 0xFFFF) << 16)
        return ((hi >> 16) + (s >> 32)) & m, s & m

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k[0], l1, h0 ^ c[3] ^ k[1], l0]
        k = [(k[0] + 0x9E3779B9) & m, (k[1] + 0xBB67AE85) & m]
    return [(w >> 8).to(torch.float64) * 2.0 ** -24 for w in c]


def exact(case, seed):
    """Path vertices in 64 bits (positions, normals, footprints); nothing for sampled values (see above)."""
    if case["kind"] != "paths":
        return None
    d = _scene(case, seed)
    x, n = d["pos"].double(), d["nrm"].double()
    P, frame = x.shape[1], LEARN_PASSES + 1
    idx = torch.arange(P, device=DEV)
    ab, found = torch.zeros(2, P, device=DEV, dtype=torch.float64), torch.zeros(P, device=DEV, dtype=torch.bool)
    for k in range(16):
        if k % 2 == 0:
            w = _philox_words(idx, frame, k // 2, seed + 5)
        t = torch.stack([2.0 * w[2 * (k % 2)] - 1.0, 2.0 * w[2 * (k % 2) + 1] - 1.0])
        hit = ~found & ((t * t).sum(0) < 1.0)
        ab = torch.where(hit, t, ab)
        found |= hit
    cos_x = torch.sqrt(torch.clamp(1.0 - (ab * ab).sum(0), min=0.0))
    t = torch.zeros_like(n)
    near = n[0].abs() < 0.9
    t[0], t[2] = near.double(), (~near).double()
    u = torch.linalg.cross(n, t, dim=0)
    u = u / u.norm(dim=0)
    v = torch.linalg.cross(n, u, dim=0)
    dr, o = ab[0] * u + ab[1] * v + cos_x * n, x + float(np.float32(1e-4)) * n
    room = torch.from_numpy(scenes.ROOM).to(DEV).double()
    tw = (torch.where(dr > 0, room[3:, None], room[:3, None]) - o) / dr
    tw = torch.where((tw > 1e-6) & (dr != 0), tw, math.inf)
    best, axis = tw.min(0)
    for b in d["boxes"].double():
        ta, tb = (b[:3, None] - o) / dr, (b[3:, None] - o) / dr
        tn, ax = torch.minimum(ta, tb).max(0)
        tf = torch.maximum(ta, tb).min(0).values
        hit = (tn < tf) & (tn > 1e-6) & (tn < best)
        best, axis = torch.where(hit, tn, best), torch.where(hit, ax, axis)
    da = dr.gather(0, axis[None])[0]
    out = torch.isinf(best)
    nrm = torch.zeros_like(n).scatter_(0, axis[None], torch.where(da > 0, -1.0, 1.0)[None].double())
    q = 100.0 * torch.clamp(cos_x, min=1e-6) * torch.clamp(da.abs(), min=1e-6)
    return [torch.where(out, o, o + torch.where(out, 0.0, best) * dr), torch.where(out, 0.0, nrm),
            torch.where(out, math.inf, best * torch.sqrt(math.pi / q)), None, None, None, None]

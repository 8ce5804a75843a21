"""Performance cases: what users of this package have it do, over its range.

Every case goes through the public Python API.  `listed()` names the fixed
cases, `draw(rng)` gives further ones of the same kinds and ranges,
`prepare(case, seed)` builds what a program holds before the call,
`run(state)` makes one pass, `work(case)` counts what a pass cannot do
without and `exact(case, seed)` gives 64-bit references where plain torch can
compute them.  Kinds of case:

  step         one loss-and-gradient evaluation of the nested SGD (whole
               images, or a stochastic pixel batch)
  autograd     differentiable rendering: render() forward and backward
  disney       the loss and gradient under the Disney material model
  cached       the loss and gradient with the radiance cache ending paths
  batch        several optimisation steps of many scenes in one batch
  rays         closest-hit ray casting
  cache_query  the cache network on given rows, with its input gradient
  cache_grad   the cache's training loss and gradients on given rows
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1903_07145_gb300 import scenes
from paper_1903_07145_gb300.batch import SceneSet
from paper_1903_07145_gb300.tracer import AdamOptions, CacheOptions, TraceOptions, Tracer, render

# Integrator settings: a program that ran the autotuner once on a large
# workload, one that ran it on a small one, and one that never did.
CONFIGS = {
    "tuned": dict(integrator="wavefront", wavefront_slots=1 << 25, trace_steps=24, bvh_width=4, sort_cells=6,
                  sort_dirs=2),
    "tuned_small": dict(integrator="megakernel"),
    "default": None,
}


# ---------------------------------------------------------------------------
# Scenes (host meshes; the same for every seed, as captured geometry is)
# ---------------------------------------------------------------------------
def _room(cuboids, sub, room_sub, views, width, height, lights=4, seed=1001):
    return dict(scene="room", cuboids=cuboids, sub=sub, room_sub=room_sub, views=views, width=width, height=height,
                lights=lights, scene_seed=seed)


ROOM_61K = _room(40, 11, 16, 8, 320, 240)


@functools.lru_cache(maxsize=4)
def _scene_of(key):
    c = dict(key)
    if c["scene"] == "cornell":
        sc = scenes.cornell_box(c["scene_seed"], c["width"], c["height"])
    elif c["scene"] == "room_516k":
        sc = scenes.room_500k(c["scene_seed"], n_views=c["views"], width=c["width"], height=c["height"])
    else:
        sc = scenes.indoor_room(c["scene_seed"], n_cuboids=c["cuboids"], cuboid_sub=c["sub"], room_sub=c["room_sub"],
                                n_lights=c["lights"], n_views=c["views"], width=c["width"], height=c["height"])
    return scenes.per_triangle(sc) if c.get("per_triangle") else sc


_SCENE_KEYS = ("scene", "cuboids", "sub", "room_sub", "views", "width", "height", "lights", "scene_seed",
               "per_triangle")


def _scene(case):
    return _scene_of(tuple((k, case[k]) for k in _SCENE_KEYS if k in case))


def _triangles(case):
    if case["scene"] == "cornell":
        return 34
    if case["scene"] == "room_516k":
        return 515728
    return 12 * case["cuboids"] * case["sub"] ** 2 + 12 * case["room_sub"] ** 2 + 2 * case["lights"]


def _pixels(case):
    return case.get("views", 1) * case["width"] * case["height"]


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the paper's stochastic pixel batch: B = 8 pixels, 128 colour samples, 1 derivative sample, L1
        dict(name="pixel_batch_cornell", kind="step", scene="cornell", scene_seed=1000, views=1, width=64, height=64,
             spp_r=128, spp_d=1, depth=3, loss="l1", pixel_batch=8, config="tuned_small", emit="lights"),
        # a larger pixel batch on a furnished room by a program that never tuned
        dict(name="pixel_batch_room", kind="step", **_room(10, 6, 6, 2, 320, 240, 2, 7), spp_r=64, spp_d=1, depth=5,
             loss="l2", pixel_batch=64, config="default", emit="all"),
        # texture refinement: every triangle its own material, gradients through autograd
        dict(name="autograd_per_triangle", kind="autograd", **_room(16, 7, 8, 1, 320, 240, 3, 21), per_triangle=True,
             spp_r=16, spp_d=16, depth=4, config="default", emit="lights"),
        # visibility probes: a handful of picks, and a volume of them
        dict(name="rays_4k", kind="rays", **ROOM_61K, n=4099, pattern="random", skip=False),
        dict(name="rays_1m", kind="rays", **ROOM_61K, n=1000003, pattern="random", skip=False),
        # one iteration on the 61k-triangle room, whole images, at the start of an optimisation
        dict(name="step_room61k", kind="step", **ROOM_61K, spp_r=32, spp_d=32, depth=5, loss="l2", pixel_batch=0,
             config="tuned", emit="all"),
        # the 516k-triangle room at its resolution, late in an optimisation
        dict(name="step_room516k", kind="step", scene="room_516k", scene_seed=1002, views=4, width=640, height=480,
             spp_r=16, spp_d=16, depth=6, loss="l2", pixel_batch=0, config="tuned", emit="lights"),
        # the paper's full material model
        dict(name="disney_room", kind="disney", **_room(24, 9, 12, 2, 320, 240, 4, 5), spp_r=16, spp_d=16, depth=4,
             loss="l2", config="tuned", emit="lights"),
        # paths cut at the second vertex by the radiance cache
        dict(name="cached_room", kind="cached", **ROOM_61K | dict(views=2), spp_r=32, spp_d=32, depth=5, loss="l2",
             b_term=1, config="tuned", emit="lights"),
        # the cache's network alone: queries with input gradients, and one training minibatch
        dict(name="cache_query_rows", kind="cache_query", n=500009),
        dict(name="cache_train_rows", kind="cache_grad", n=153623),
        # serving: 64 small scenes optimised together, parameters read every few steps
        dict(name="batch_cornell64", kind="batch", members=64, steps=8, spp_r=64, spp_d=1, depth=3, pixel_batch=64,
             config="tuned_small"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "pixel_batch", "pixel_batch", "autograd", "disney", "cached", "batch", "rays",
                       "rays", "cache_query", "cache_grad"])
    if kind in ("cache_query", "cache_grad"):
        return dict(kind=kind, n=_log(rng, 300, 600000))
    if kind == "batch":
        b = _log(rng, 8, 128)
        return dict(kind=kind, members=_log(rng, 4, 64), steps=rng.randint(2, 8), spp_r=rng.choice([16, 64, 100]),
                    spp_d=rng.choice([1, 2]), depth=rng.randint(2, 4), pixel_batch=b,
                    config=rng.choice(["tuned_small", "default"]))
    if rng.random() < 0.25:
        geo = dict(scene="cornell", scene_seed=rng.randint(1, 9999), views=1, width=rng.randint(24, 160),
                   height=rng.randint(24, 160))
    else:
        geo = _room(rng.randint(6, 16), _log(rng, 2, 18), rng.randint(2, 16), rng.randint(1, 3),
                    rng.choice([160, 213, 320, 401]), rng.choice([97, 120, 240, 301]), rng.randint(1, 6),
                    rng.randint(1, 9999))
    emit = rng.choice(["all", "lights"])
    if kind == "rays":
        return dict(kind=kind, **geo, n=_log(rng, 500, 2000000), pattern=rng.choice(["random", "camera"]),
                    skip=rng.random() < 0.3)
    opts = dict(depth=rng.randint(1, 6), emit=emit)
    if kind == "pixel_batch":
        return dict(kind="step", **geo, **opts, spp_r=rng.choice([16, 33, 64, 128, 256]), spp_d=rng.choice([1, 1, 2]),
                    loss=rng.choice(["l1", "l2"]), pixel_batch=_log(rng, 4, 2048),
                    config=rng.choice(["tuned_small", "default"]))
    opts |= dict(spp_r=rng.choice([4, 7, 16, 32]), spp_d=rng.choice([4, 7, 16]))
    if kind == "autograd":
        return dict(kind=kind, **geo, **opts, per_triangle=rng.random() < 0.4 and geo["scene"] == "room",
                    config=rng.choice(["tuned", "default"]))
    opts |= dict(loss=rng.choice(["l1", "l2"]), config=rng.choice(["tuned", "default"]))
    if kind == "cached":
        opts["depth"] = rng.randint(3, 6)
        return dict(kind=kind, **geo, **opts, b_term=rng.choice([1, 2]))
    if kind == "disney":
        return dict(kind=kind, **geo, **opts)
    return dict(kind="step", **geo, **opts, pixel_batch=0)


# ---------------------------------------------------------------------------
# Preparation
# ---------------------------------------------------------------------------
def _options(case):
    return TraceOptions(spp_r=case["spp_r"], spp_d=case["spp_d"], max_depth=case["depth"],
                        loss=case.get("loss", "l2"), pixel_batch=case.get("pixel_batch", 0))


def _estimate(scene, seed, emit):
    """The unknowns mid-way: around one half at the start of an optimisation
    (every segment still emits), around the truth late in one."""
    rng = np.random.default_rng(seed)
    if emit == "all":
        p = 0.5 * rng.uniform(0.9, 1.1, (scene.n_segments, 10))
    else:
        p = np.asarray(scene.gt_params, np.float64) * rng.uniform(0.8, 1.2, (scene.n_segments, 10))
        p[:, 6] = np.clip(p[:, 6], 0.05, 1.0)
    return p.astype(np.float32)


def _pictures(pixels, seed):
    """Captured images: smooth radiance with per-pixel noise."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.arange(pixels, device="cuda", dtype=torch.float32)[:, None]
    f = 0.01 + 0.04 * torch.rand(3, device="cuda", generator=g)
    noise = torch.rand((pixels, 3), device="cuda", generator=g)
    return 0.6 + 0.4 * torch.sin(x * f) + 0.4 * noise


def _tracer(case, seed):
    tr = Tracer(_scene(case), seed=seed)
    if CONFIGS[case.get("config", "default")] is not None:
        tr.configure(**CONFIGS[case["config"]])
    return tr


def _rays(case, seed):
    sc = _scene(case)
    n = case["n"]
    if case["pattern"] == "random":
        o, d = scenes.random_rays(sc, n, seed)
    else:  # a pinhole camera's grid of rays, row by row
        rng = np.random.default_rng(seed)
        m = np.asarray(sc.cameras[0].cam_to_world, np.float64).reshape(3, 4)
        w = max(1, int(math.sqrt(n * 4 / 3)))
        i = np.arange(n)
        local = np.stack([(i % w + rng.random(n)) / w - 0.5, 0.375 - (i // w + rng.random(n)) / w, -np.ones(n)], 1)
        d = local @ m[:, :3].T
        d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
        o = np.broadcast_to(m[:, 3], (n, 3)).astype(np.float32)
    skip = None
    if case["skip"]:
        skip = np.random.default_rng(seed + 1).integers(-1, sc.n_tri, n).astype(np.int32)
    return o, d, skip


def _cache_rows(case, seed):
    """Rows of the cache's network: positions on a few surfaces of the unit
    cube (where paths end), unit directions and normals, materials, targets."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = case["n"]
    r = lambda *s: torch.rand(s, device="cuda", generator=g)  # noqa: E731
    x = r(n, 3)
    axis = torch.randint(0, 3, (n, 1), device="cuda", generator=g)
    plane = torch.randint(0, 6, (n, 1), device="cuda", generator=g).float() / 5.0
    x.scatter_(1, axis, plane)
    unit = lambda v: v / v.norm(dim=1, keepdim=True)  # noqa: E731
    d = unit(torch.randn((n, 3), device="cuda", generator=g))
    nrm = torch.zeros((n, 3), device="cuda").scatter_(1, axis, 1.0)
    p7 = torch.cat([0.1 + 0.8 * r(n, 3), 0.3 * r(n, 3), 0.05 + 0.75 * r(n, 1)], 1)
    return x, d, nrm, p7, r(n, 3) * 2.0


_WEIGHT_SHAPES = ((80, 64), (64, 64), (64, 64), (64, 64), (64, 16))


def _cache_state(seed):
    """Weights at the usual initial scale and a trained-looking hash table."""
    rng = np.random.default_rng(seed + 77)
    w = np.concatenate([rng.uniform(-1, 1, s).ravel() * math.sqrt(6.0 / s[0]) for s in _WEIGHT_SHAPES])
    t = rng.random(16 * 524288 * 2, dtype=np.float32) - np.float32(0.5)
    return w.astype(np.float32), t


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        members = [scenes.cornell_variant(k) for k in range(case["members"])]
        ss = SceneSet(members, seed=seed)
        if CONFIGS[case["config"]] is not None:
            ss.configure(**CONFIGS[case["config"]])
        for i, sc in enumerate(members):
            p = _estimate(sc, seed + i, "lights")
            free = np.zeros((sc.n_segments, 10), np.uint8)
            free[:, 0:3] = free[:, 7:10] = 1
            ss.set_params(i, p, free)
            ss.set_targets(i, _pictures(ss.n_pix[i], seed + i))
        ss.make_batch()
        return dict(kind=kind, set=ss, opts=_options(case), adam=AdamOptions(), steps=case["steps"])
    if kind in ("cache_query", "cache_grad"):
        tr = Tracer(scenes.cornell_box(1000), seed=seed)
        tr.configure_cache(CacheOptions())
        tr.set_cache_weights(*_cache_state(seed))
        x, d, nrm, p7, y = _cache_rows(case, seed)
        return dict(kind=kind, tracer=tr, rows=(x, d, nrm, p7), extra=y)
    tr = _tracer(case, seed)
    if kind == "rays":
        o, d, skip = _rays(case, seed)
        dev = lambda a: None if a is None else torch.from_numpy(a).cuda()  # noqa: E731
        return dict(kind=kind, tracer=tr, rays=(dev(o), dev(d), dev(skip)))
    sc = _scene(case)
    state = dict(kind=kind, tracer=tr, opts=_options(case), iteration=seed % 1000)
    p = _estimate(sc, seed, case["emit"])
    if kind == "autograd":
        state["params"] = torch.from_numpy(p).cuda().requires_grad_(True)
        state["target"] = _pictures(tr.n_pix, seed)
        return state
    tr.set_targets(_pictures(tr.n_pix, seed))
    if kind == "disney":
        q = scenes.disney_materials(sc, seed)
        if case["emit"] == "all":
            q[:, 13:16] = p[:, 7:10]
        tr.disney_set_params(q)
        return state
    tr.set_params(p)
    if kind == "cached":
        tr.configure_cache(CacheOptions(b_term=case["b_term"]))
        tr.set_cache_weights(*_cache_state(seed))
    return state


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "batch":
        ss = state["set"]
        # the losses are logged in the precision of the radiances they sum
        losses = [ss.batch_step(state["opts"], state["adam"]).astype(np.float32) for _ in range(state["steps"])]
        return np.stack(losses), np.concatenate([ss.batch_params(i) for i in range(len(ss.sids))])
    tr = state["tracer"]
    if kind == "rays":
        return tr.trace_rays(*state["rays"])
    if kind == "cache_query":
        return tr.cache_eval(*state["rows"], upstream=state["extra"])
    if kind == "cache_grad":
        return tr.cache_grad(*state["rows"], target=state["extra"])
    if kind == "autograd":
        img = render(state["params"], tr, state["opts"], iteration=state["iteration"])
        loss = (img - state["target"]).square().mean()
        (grad,) = torch.autograd.grad(loss, state["params"])
        return img.detach(), grad
    if kind == "disney":
        return tr.disney_loss_grad(state["opts"], state["iteration"])
    return tr.loss_grad(state["opts"], state["iteration"])


# ---------------------------------------------------------------------------
# Necessary work
# ---------------------------------------------------------------------------
def work(case):
    """Inputs read once and outputs written once; operations of the shortest
    traversal (one box test per tree level and two triangle tests a ray) and
    of the materials at each vertex."""
    kind = case["kind"]
    if kind in ("cache_query", "cache_grad"):
        n, macs = case["n"], sum(a * b for a, b in _WEIGHT_SHAPES)
        table = 16 * 524288 * 2 * 4
        touched = min(table, n * 16 * 8 * 8)
        if kind == "cache_query":
            return dict(bytes=n * (12 * 4 + 28 + 12 + 28) + touched, flops=n * 4 * macs)
        return dict(bytes=n * (12 * 4 + 28) + touched + table, flops=n * 6 * macs)

    def trace(rays, tris):
        return rays * (24.0 * math.log2(max(tris, 2)) + 2 * 50.0)

    if kind == "rays":
        t = _triangles(case)
        return dict(bytes=t * 40 + case["n"] * (24 + 16 + (4 if case["skip"] else 0)), flops=trace(case["n"], t))
    if kind == "batch":
        paths = case["members"] * case["pixel_batch"] * (case["spp_r"] + case["spp_d"]) * case["steps"]
        rays = paths * (2 * case["depth"] + 1)
        return dict(bytes=case["members"] * case["steps"] * (case["pixel_batch"] * 12 + 34 * 40 + 7 * 40 * 4),
                    flops=trace(rays, 34) + 200.0 * rays)
    t, pix = _triangles(case), case.get("pixel_batch", 0) or _pixels(case)
    depth_r = min(case["depth"], case["b_term"]) if kind == "cached" else case["depth"]
    rays = pix * (case["spp_r"] + case["spp_d"]) * (2 * depth_r + 1)
    segs = t if case.get("per_triangle") else 60
    flops = trace(rays, t) + 200.0 * rays
    if kind == "cached":
        flops += pix * (2 * case["spp_r"] + 4 * case["spp_d"]) * sum(a * b for a, b in _WEIGHT_SHAPES)
    return dict(bytes=t * 40 + pix * 24 + segs * 80, flops=flops)


# ---------------------------------------------------------------------------
# 64-bit references
# ---------------------------------------------------------------------------
def _exact_rays(case, seed):
    sc = _scene(case)
    if case["n"] * sc.n_tri > 4e8:
        return None
    o, d, skip = (None if a is None else torch.from_numpy(a).cuda() for a in _rays(case, seed))
    o, d = o.double(), d.double()
    p = torch.from_numpy(np.asarray(sc.positions, np.float32)[np.asarray(sc.indices, np.int64)]).cuda().double()
    a, e1, e2 = p[:, 0], p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]
    ids = torch.arange(sc.n_tri, device="cuda")
    outs = []
    step = max(1, int(2e7 // sc.n_tri))
    for i in range(0, case["n"], step):
        oo, dd = o[i:i + step, None], d[i:i + step, None]
        h = torch.cross(dd.expand(-1, sc.n_tri, -1), e2.expand(dd.shape[0], -1, -1), dim=2)
        det = (h * e1).sum(2)
        s = oo - a
        u = (s * h).sum(2) / det
        q = torch.cross(s, e1.expand_as(s), dim=2)
        v = (dd * q).sum(2) / det
        t = (e2 * q).sum(2) / det
        hit = (u >= 0) & (v >= 0) & (u + v <= 1) & (t > 0)
        if skip is not None:
            hit &= ids != skip[i:i + step, None]
        t = torch.where(hit, t, torch.inf)
        k = t.argmin(1, keepdim=True)
        best = t.gather(1, k)
        miss = torch.isinf(best)
        zero = torch.zeros_like(best)
        outs.append(torch.cat([best, torch.where(miss, zero, u.gather(1, k)), torch.where(miss, zero, v.gather(1, k))], 1))
    r = torch.cat(outs)
    return None, r[:, 0].contiguous(), r[:, 1].contiguous(), r[:, 2].contiguous()


def _encode(table, x):
    """Multiresolution hash encoding of positions in the unit cube."""
    b = math.exp((math.log(2048.0) - math.log(16.0)) / 15)
    feats = []
    for level in range(16):
        n = int(math.floor(16 * b ** level))
        p = x * n
        c0 = p.floor()
        f = p - c0
        c0 = c0.long()
        acc = 0.0
        for k in range(8):
            bit = torch.tensor([k & 1, (k >> 1) & 1, k >> 2], device=x.device)
            c = (c0 + bit).clamp(max=n)
            w = torch.where(bit.bool(), f, 1.0 - f).prod(1, keepdim=True)
            if (n + 1) ** 3 <= 524288:
                h = c[:, 0] + c[:, 1] * (n + 1) + c[:, 2] * (n + 1) ** 2
            else:
                h = c[:, 0] ^ (c[:, 1] * 2654435761 & 0xFFFFFFFF) ^ (c[:, 2] * 805459861 & 0xFFFFFFFF)
            acc = acc + w * table[level, h & 524287]
        feats.append(acc)
    return torch.cat(feats, 1)


def _harmonics(d):
    """Real spherical harmonics of degrees 0 to 3."""
    x, y, z = d.unbind(1)
    a, b = math.sqrt(3 / (4 * math.pi)), math.sqrt(15 / math.pi) / 2
    c, e = math.sqrt(5 / math.pi) / 4, math.sqrt(35 / (2 * math.pi)) / 4
    f, g = math.sqrt(21 / (2 * math.pi)) / 4, math.sqrt(7 / math.pi) / 4
    k = math.sqrt(105 / math.pi)
    return torch.stack([
        torch.full_like(x, 0.5 / math.sqrt(math.pi)), -a * y, a * z, -a * x, b * x * y, -b * y * z,
        c * (3 * z * z - 1), -b * x * z, b / 2 * (x * x - y * y), -e * y * (3 * x * x - y * y), k / 2 * x * y * z,
        -f * y * (5 * z * z - 1), g * z * (5 * z * z - 3), -f * x * (5 * z * z - 1), k / 4 * z * (x * x - y * y),
        -e * x * (x * x - 3 * y * y)], 1)


def _exact_cache(case, seed):
    w, t = _cache_state(seed)
    x, d, nrm, p7, y = (v.double() for v in _cache_rows(case, seed))
    query = case["kind"] == "cache_query"
    # a hidden unit at its kink may be decided the other way in BF16, which
    # moves that row's input gradient by a jump: only many rows average it out
    many = case["n"] >= 20000
    table = torch.from_numpy(t).cuda().double().reshape(16, 524288, 2).requires_grad_(not query)
    flat = torch.from_numpy(w).cuda().double().requires_grad_(not query)
    p7.requires_grad_(query)
    h = torch.cat([_encode(table, x), _harmonics(d), _harmonics(nrm), p7, x.new_zeros(x.shape[0], 9)], 1)
    at = 0
    for i, (a, b) in enumerate(_WEIGHT_SHAPES):
        h = h @ flat[at:at + a * b].reshape(a, b)
        h = h.relu() if i < 4 else h[:, :3]
        at += a * b
    if query:
        (g,) = torch.autograd.grad((h * y).sum(), p7)
        return h.detach(), g if many else None
    loss = ((h - y).square() / (h.detach().square() + 0.01)).mean()
    gw, gt = torch.autograd.grad(loss, (flat, table))
    return float(loss.detach()), gw, gt.reshape(-1) if many else None


def exact(case, seed):
    if case["kind"] == "rays":
        return _exact_rays(case, seed)
    if case["kind"] in ("cache_query", "cache_grad"):
        return _exact_cache(case, seed)
    return None  # Monte Carlo transport: no 64-bit value without tracing the same paths

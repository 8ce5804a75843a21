"""Every BVH form gives the same hits: binary, 4-wide (8-bit boxes, or planes
on the scene grid where the builder picks it) and 8-wide, on meshes where the
forms differ most: coincident triangles (exact ties), a flat sheet, a small
detail in a large scene (keeps the 8-bit boxes), one and two triangles."""
import numpy as np
import pytest
import torch

from paper_1903_07145_gb300 import scenes
from paper_1903_07145_gb300.scenes import Scene
from paper_1903_07145_gb300.tracer import TraceOptions, Tracer

pytestmark = pytest.mark.gpu


def _mesh(pos, seed=0):
    pos = np.asarray(pos, np.float32).reshape(-1, 3, 3)
    n = len(pos)
    cam = scenes.look_camera(pos.mean((0, 1)) + np.array([0, 0, 3 * np.ptp(pos) / 2]), 0.0, 0.0, 60.0, 24, 20)
    gt = np.full((2, 10), 0.4, np.float32)
    return Scene("mesh", pos.reshape(-1, 3), np.arange(3 * n, dtype=np.uint32).reshape(n, 3),
                 (np.arange(n) % 2).astype(np.uint32), 2, [cam], gt)


def _soup(n, size=0.2, scale=1.0):
    rng = np.random.default_rng(n)
    return scale * (rng.uniform(-2, 2, (n, 1, 3)) + rng.uniform(-size, size, (n, 3, 3)))


def _forms():
    soup = _soup(600)
    sheet = _soup(500)
    sheet[..., 1] = 0.25
    return {
        "ties": np.concatenate([soup, soup, soup[::-1]]),
        "flat": sheet,
        "detail": np.concatenate([_soup(2000, 0.3, 1e-3), [[[-40, -40, -40], [-41, -40, -40], [-40, -41, -41]],
                                                            [[40, 40, 40], [41, 40, 40], [40, 41, 41]]]]),
        "one": _soup(1),
        "two": _soup(2),
    }


@pytest.mark.parametrize("name", ["ties", "flat", "detail", "one", "two"])
def test_bvh_forms_give_the_same_hits(name):
    pos = _forms()[name].astype(np.float32)
    sc = _mesh(pos)
    tr = Tracer(sc, seed=1)
    tr.set_params(sc.gt_params)
    rng = np.random.default_rng(3)
    n = 20011
    # towards points on the triangles, and along the axes through them
    tri = pos[rng.integers(0, len(pos), n)].astype(np.float64)
    w = rng.dirichlet((1, 1, 1), n)
    target = (tri * w[:, :, None]).sum(1)
    o = target + rng.normal(size=(n, 3)) * rng.choice([1e-2, 1.0, 100.0], (n, 1))
    d = target - o
    ax = rng.integers(0, 3, n)
    axis = rng.random(n) < 0.2
    d[axis] = np.eye(3)[ax[axis]] * np.where(rng.random(axis.sum()) < 0.5, -1, 1)[:, None]
    o[axis] = target[axis] - 2.0 * d[axis]
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    o, d = (torch.from_numpy(a.astype(np.float32)).cuda() for a in (o, d))
    opts = TraceOptions(spp_r=4, max_depth=2)
    ref = img = None
    for width in (2, 4, 8):
        tr.configure(bvh_width=width)
        got = [v.cpu() for v in tr.trace_rays(o, d)]
        pic = tr.render(opts).cpu()
        if ref is None:
            ref, img = got, pic
            assert (ref[0] >= 0).float().mean() > 0.5
        for a, b in zip(ref, got):
            assert torch.equal(a, b), f"width {width}"
        assert torch.equal(img, pic), f"width {width}"
    if name == "ties":  # the smallest id of the coincident copies
        hit = ref[0][ref[0] >= 0].numpy()
        assert (hit < 600).all()
    tr.close()


@pytest.mark.parametrize("n", [1, 31, 4863, 4865, 155647, 155649, 400001])
def test_ray_counts_around_the_launch_forms(n):
    """A launch with at most as many rays as lanes spreads them over its warps,
    a larger one refills: the same hits for a ray wherever it stands, with and
    without skipped triangles, and twice in a row (the counters are cleared)."""
    sc = scenes.indoor_room(3, n_cuboids=6, cuboid_sub=4, room_sub=4, n_lights=2, n_views=1, width=8, height=8)
    tr = Tracer(sc, seed=1)
    o, d = scenes.random_rays(sc, 997, 4)
    skip = np.random.default_rng(5).integers(-1, sc.n_tri, 997).astype(np.int32)
    pick = torch.from_numpy(np.random.default_rng(n).integers(0, 997, n))
    o, d, skip = (torch.from_numpy(a) for a in (o, d, skip))
    for sk in (None, skip):
        ref = [v.cpu() for v in tr.trace_rays(o, d, sk)]
        for _ in range(2):
            got = [v.cpu() for v in tr.trace_rays(o[pick], d[pick], None if sk is None else sk[pick])]
            for a, b in zip(ref, got):
                assert torch.equal(a[pick], b)
    tr.close()


def test_a_captured_launch_keeps_no_counter():
    """More rays than a wave has lanes, captured: graphs replayed side by side
    and beside an eager call give each its own hits."""
    sc = scenes.indoor_room(3, n_cuboids=6, cuboid_sub=4, room_sub=4, n_lights=2, n_views=1, width=8, height=8)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        tr = Tracer(sc, seed=1)
        rays = [[torch.from_numpy(a).cuda() for a in scenes.random_rays(sc, 200003, k)] for k in (4, 5)]
        ref = [[v.clone() for v in tr.trace_rays(*r)] for r in rays]
        stream.synchronize()
        graphs, outs = [], []
        for r in rays:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                outs.append(tr.trace_rays(*r))
            graphs.append(g)
        torch.cuda.synchronize()
    other = torch.cuda.Stream()
    for _ in range(3):
        with torch.cuda.stream(stream):
            graphs[0].replay()
            eager = tr.trace_rays(*rays[1])
        with torch.cuda.stream(other):
            graphs[1].replay()
        torch.cuda.synchronize()
        for got, want in ((outs[0], ref[0]), (outs[1], ref[1]), (eager, ref[1])):
            for a, b in zip(got, want):
                assert torch.equal(a, b)
    tr.close()

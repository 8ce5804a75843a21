"""Launches on either side of the limits at which their form changes, the
limits taken from the device: derivative passes of one path a thread (14 warps
of paths an SM; more: a pixel's paths share a warp's lanes), and ray casting
in one wave or more."""
import time

import numpy as np
import pytest
import torch

from paper_1903_07145_gb300 import scenes
from paper_1903_07145_gb300.batch import SceneSet
from paper_1903_07145_gb300.tracer import AdamOptions, TraceOptions, Tracer

pytestmark = pytest.mark.gpu
SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152


def _room():
    return scenes.indoor_room(9, n_cuboids=4, cuboid_sub=2, room_sub=2, n_lights=2, n_views=2, width=40, height=31)


def _tracer(integrator, sc):
    tr = Tracer(sc, seed=4)
    if integrator != "unset":
        tr.configure(integrator)
    tr.set_params(sc.gt_params)
    tr.set_targets(np.random.default_rng(2).random((tr.n_pix, 3)).astype(np.float32))
    return tr


def _sizes():
    out = []
    for warps in (8, 14):
        paths = 32 * warps * SMS
        out += [(paths - 1, 1), (paths, 1), (paths + 1, 1), (paths // 129, 129), (paths // 129 + 1, 129),
                (paths // 7 + 1, 7), (paths // 32, 32), (paths // 32 + 1, 32)]
    return out


@pytest.mark.parametrize("sub", [0, 6, 9])
def test_derivative_passes_around_the_limits(sub):
    """Gradients agree with the wavefront's to the rounding of FP32 sums in
    another order (rel 1e-5), with accumulators in shared memory (few segments,
    and a segment per triangle) and in global memory (above 5120 segments)."""
    sc = _room()
    if sub:
        sc = scenes.per_triangle(scenes.indoor_room(9, n_cuboids=6, cuboid_sub=sub, room_sub=4, n_lights=2, n_views=2,
                                                    width=40, height=31))
        assert (sc.n_segments > 5120) == (sub == 9)
    tracers = {k: _tracer(k, sc) for k in ("wavefront", "megakernel", "unset")}
    for batch, spp_d in _sizes():
        opts = TraceOptions(spp_r=1, spp_d=spp_d, max_depth=3, pixel_batch=batch)
        want = tracers["wavefront"].loss_grad(opts, 5)[1].double()
        for k in ("megakernel", "unset"):
            got = tracers[k].loss_grad(opts, 5)[1].double()
            assert (got - want).norm() <= 1e-5 * want.norm(), (k, batch, spp_d)
    for tr in tracers.values():
        tr.close()


def _best(f, n=5):
    f()
    out = []
    for _ in range(n):
        torch.cuda.synchronize()
        t = time.perf_counter()
        f()
        torch.cuda.synchronize()
        out.append(time.perf_counter() - t)
    return min(out)


@pytest.mark.parametrize("spp_d", [7, 33, 129])
def test_no_pass_runs_a_pixels_paths_one_after_the_other(spp_d):
    """A program that sets no integrator is not slower than one that sets the
    wavefront (which it is quicker than by a half) where a pixel's paths do
    not divide into lanes: a serial pixel is 2 to 30 times as slow."""
    opts = TraceOptions(spp_r=1, spp_d=spp_d, max_depth=5, pixel_batch=32 * 12 * SMS // spp_d)
    took = {}
    for k in ("wavefront", "unset"):
        tr = _tracer(k, _room())
        took[k] = _best(lambda: tr.loss_grad(opts, 1))
        tr.close()
    assert took["unset"] <= 1.2 * took["wavefront"], took


def test_a_batchs_derivative_pass_around_the_limits():
    """The first step's gradient, through the parameters it leads to: Adam's
    first step is lr times the gradient's sign where it is not noise."""
    members = [scenes.cornell_variant(k) for k in range(3)]
    for per_member, spp_d in [(32 * 14 * SMS // 3 // 129, 129), (32 * 14 * SMS // 3 // 129 + 1, 129), (32 * 9 * SMS // 3, 1)]:
        opts = TraceOptions(spp_r=1, spp_d=spp_d, max_depth=3, pixel_batch=per_member)
        params = {}
        for integrator in ("wavefront", "megakernel", "unset"):
            ss = SceneSet(members, seed=6)
            if integrator != "unset":
                ss.configure(integrator)
            for i, sc in enumerate(members):
                free = np.zeros((sc.n_segments, 10), np.uint8)
                free[:, 0:3] = 1
                ss.set_params(i, sc.gt_params, free)
                ss.set_targets(i, torch.from_numpy(np.random.default_rng(i).random((ss.n_pix[i], 3))))
            ss.make_batch()
            ss.batch_step(opts, AdamOptions())
            params[integrator] = np.concatenate([ss.batch_params(i) for i in range(3)])
            ss.close()
        for k in ("megakernel", "unset"):
            close = np.abs(params[k] - params["wavefront"]) < 1e-5
            assert close.mean() >= 0.98, (k, per_member, spp_d)


@pytest.mark.parametrize("blocks", [1, 3])
def test_ray_counts_around_one_wave(blocks):
    """`blocks` blocks of four warps an SM: one ray a warp, one wave of lanes
    (more rays are fetched), each with one ray fewer and one more."""
    sc = scenes.indoor_room(3, n_cuboids=6, cuboid_sub=4, room_sub=4, n_lights=2, n_views=1, width=8, height=8)
    tr = Tracer(sc, seed=1)
    o, d = (torch.from_numpy(a).cuda() for a in scenes.random_rays(sc, 997, 4))
    ref = tr.trace_rays(o, d)
    tr.configure(blocks_per_sm=blocks)
    for limit in (4 * blocks * SMS, 128 * blocks * SMS):
        for n in (limit - 1, limit, limit + 1, 2 * limit + 1):
            pick = torch.from_numpy(np.random.default_rng(n).integers(0, 997, n)).cuda()
            for a, b in zip(ref, tr.trace_rays(o[pick], d[pick])):
                assert torch.equal(a[pick], b), n
    tr.close()

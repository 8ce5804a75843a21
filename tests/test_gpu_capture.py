"""Calls under stream capture: a replayed graph repeats the captured call,
whatever the context ran in between.  Images are equal bit for bit; gradients
agree to the rounding of FP32 sums in another order (rel 1e-5)."""
import contextlib
import ctypes as C

import numpy as np
import pytest
import torch

from paper_1903_07145_gb300 import _lib as L
from paper_1903_07145_gb300 import scenes
from paper_1903_07145_gb300.tracer import CacheOptions, TraceOptions, Tracer

pytestmark = pytest.mark.gpu
MODES = ["unset", "wavefront", "megakernel"]  # unset: the integrator by the size of the pass
OPTS = TraceOptions(spp_r=9, spp_d=3, max_depth=3)
PICKS = TraceOptions(spp_r=9, spp_d=3, max_depth=3, pixel_batch=33)


def _room():
    return scenes.indoor_room(9, n_cuboids=4, cuboid_sub=2, room_sub=2, n_lights=2, n_views=2, width=40, height=31)


def _loss_grad(tr, opts, iteration, disney=False):
    """The call without its loss, which would wait for the stream."""
    out = torch.empty((tr.n_seg, 16 if disney else 10), device="cuda")
    f = L.ipt_disney_loss_grad if disney else L.ipt_loss_grad
    f(tr.ctx, tr.sid, opts.c(), iteration, False, out.data_ptr())
    return out


CALLS = {
    "render": lambda tr, w: tr.render(OPTS, view=1, iteration=2),
    "backward": lambda tr, w: tr.backward(w, OPTS, iteration=2),
    "loss_grad": lambda tr, w: _loss_grad(tr, OPTS, 2),
    "pixel_batch": lambda tr, w: _loss_grad(tr, PICKS, 2),
    "disney_render": lambda tr, w: tr.disney_render(OPTS, view=1, iteration=2),
    "disney_pixel_batch": lambda tr, w: _loss_grad(tr, PICKS, 2, disney=True),
}


def _tracer(mode, seed=4):
    sc = _room()
    tr = Tracer(sc, seed=seed)
    if mode != "unset":
        tr.configure(mode)
    tr.set_params(sc.gt_params)
    tr.disney_set_params(scenes.disney_materials(sc, 3))
    rng = np.random.default_rng(2)
    tr.set_targets(rng.random((tr.n_pix, 3)).astype(np.float32))
    return tr, torch.from_numpy(rng.normal(size=(tr.n_pix, 3)).astype(np.float32)).cuda()


def _same(name, got, want):
    if "render" in name:
        return torch.equal(got, want)
    return (got.double() - want.double()).norm() <= 1e-5 * want.double().norm()


@pytest.mark.parametrize("mode", MODES)
def test_replays_repeat_the_call(mode):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        tr, w = _tracer(mode)
        want = {k: f(tr, w).clone() for k, f in CALLS.items()}
        stream.synchronize()
        graphs, got = {}, {}
        for k, f in CALLS.items():
            graphs[k] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graphs[k], stream=stream):
                got[k] = f(tr, w)
        for k in CALLS:
            # another view, other entries: whatever a replay shares with later calls is theirs by now
            tr.render(OPTS, view=0, iteration=5)
            _loss_grad(tr, PICKS, 7)
            got[k].fill_(float("nan"))
            graphs[k].replay()
            assert _same(k, got[k], want[k]), k
        tr.synchronize()
        tr.close()


SMALL, LARGE = TraceOptions(spp_r=1, spp_d=1, max_depth=3), TraceOptions(spp_r=256, spp_d=128, max_depth=6)


@pytest.mark.parametrize("warm", ["same", "smaller", "none"])
def test_a_capture_allocates_what_its_pass_needs(warm):
    """A program that set no integrator captures passes on either side of the
    size rule, warmed up by the same pass, by a smaller one on the other
    integrator, or not at all."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ref, w = _tracer("unset")
        for opts in (SMALL, OPTS, LARGE):
            want = ref.render(opts), ref.backward(w, opts)
            tr, _ = _tracer("unset")
            if warm != "none":
                tr.render(opts if warm == "same" else SMALL), tr.backward(w, opts if warm == "same" else SMALL)
            stream.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                got = tr.render(opts), tr.backward(w, opts)
            first = [v.clone() for v in (tr.render(SMALL), tr.backward(w, SMALL))]
            # what a larger call allocates afterwards leaves the graph its buffers
            tr.render(LARGE, iteration=4), tr.backward(w, LARGE, iteration=4)
            for v in got:
                v.fill_(float("nan"))
            for _ in range(2):
                g.replay()
                assert _same("render", got[0], want[0]) and _same("backward", got[1], want[1])
            again = tr.render(SMALL), tr.backward(w, SMALL)
            assert _same("render", again[0], first[0]) and _same("backward", again[1], first[1])
            tr.synchronize()
            tr.close()
        ref.close()


def test_tables_follow_the_parameters_through_replays():
    """A call uses the parameters it is given, or the scene's at that time,
    whatever the calls around it (eager or replayed) built tables from."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        tr, _ = _tracer("wavefront")
        sc = tr.scene
        rng = np.random.default_rng(8)
        own, new, other = (np.asarray(sc.gt_params * s, np.float32) for s in (1.0, 0.7, 0.4))
        given = torch.from_numpy(other).cuda()
        mats = [scenes.disney_materials(sc, k) for k in (3, 5)]
        spare = torch.from_numpy(scenes.disney_materials(sc, 9)).cuda()
        r = lambda **k: tr.render(OPTS, **k).clone()  # noqa: E731
        d = lambda **k: tr.disney_render(OPTS, **k).clone()  # noqa: E731
        want = {}
        for name, p, m in (("new", new, mats[1]), ("own", own, mats[0])):
            tr.set_params(p), tr.disney_set_params(m)
            want[name] = r(), r(params=given), d(), d(sampling_params=spare)
        stream.synchronize()
        g = [torch.cuda.CUDAGraph() for _ in range(4)]
        outs = []
        for graph, f in zip(g, (lambda: tr.render(OPTS), lambda: tr.render(OPTS, params=given),
                                lambda: tr.disney_render(OPTS),
                                lambda: tr.disney_render(OPTS, sampling_params=spare))):
            with torch.cuda.graph(graph, stream=stream):
                outs.append(f())
        for name in ("own", "new"):
            if name == "new":
                tr.set_params(new), tr.disney_set_params(mats[1])
            for order in rng.permuted(np.tile(np.arange(4), (6, 1)), axis=1):
                for k in order:
                    g[k].replay()
                    assert torch.equal(outs[k], want[name][k])
                    assert torch.equal(r(), want[name][0]) and torch.equal(d(), want[name][2])
                    r(params=given), d(sampling_params=spare)
        tr.synchronize()
        tr.close()


@pytest.mark.parametrize("mode", MODES)
def test_a_graph_keeps_buffers_that_are_outgrown(mode):
    """Pixel batches (both models) and, on the wavefront, cached passes: the
    entries' and queries' buffers of a graph outlive their growth."""
    big = TraceOptions(spp_r=2, spp_d=2, max_depth=3, pixel_batch=5000)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        tr, w = _tracer(mode)
        calls = ["pixel_batch", "disney_pixel_batch"]
        want = {k: CALLS[k](tr, w).clone() for k in calls}
        if mode == "wavefront":
            tr.configure(mode, wavefront_slots=4096)
            tr.configure_cache(CacheOptions())
            calls.append("render")
            want["render"] = CALLS["render"](tr, w).clone()
            tr.configure_cache(CacheOptions(enabled=False))
            plain = CALLS["render"](tr, w)
            assert not torch.equal(plain, want["render"])
        stream.synchronize()
        graphs, got = {}, {}
        for k in calls:
            if k == "render":
                tr.configure_cache(CacheOptions())
                CALLS[k](tr, w)
                stream.synchronize()
            graphs[k] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graphs[k], stream=stream):
                got[k] = CALLS[k](tr, w)
        if mode == "wavefront":  # larger buffers for the queries and the path state
            tr.configure(mode, wavefront_slots=8192)
            CALLS["render"](tr, w)
            tr.configure_cache(CacheOptions(enabled=False))
        _loss_grad(tr, big, 5), _loss_grad(tr, big, 5, disney=True)
        stream.synchronize()
        spare = [torch.full((1 << 16,), float("nan"), device="cuda") for _ in range(64)]  # in freed memory, if any
        for k in calls:
            got[k].fill_(float("nan"))
            graphs[k].replay()
            assert _same(k, got[k], want[k]), k
        tr.synchronize()
        del spare
        tr.close()


@contextlib.contextmanager
def _lost_capture(stream):
    """A capture that a call inside invalidates (by the driver's calls: torch's
    own bookkeeping would outlive the failure)."""
    cu = C.CDLL("libcuda.so.1")
    graph = C.c_void_p()
    torch.cuda.synchronize()
    assert cu.cuStreamBeginCapture_v2(C.c_void_p(stream.cuda_stream), 2) == 0
    yield
    assert cu.cuStreamEndCapture(C.c_void_p(stream.cuda_stream), C.byref(graph)) != 0


def test_a_read_that_cannot_wait_leaves_its_output():
    """A call that returns host data fails under capture; it does not hand out
    what an earlier call read."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        tr, _ = _tracer("wavefront")
        before = tr.get_params()
        assert np.isfinite(before).all()
        out = np.full_like(before, np.nan)
        with _lost_capture(stream), pytest.raises(L.IptError):
            L.ipt_params_get(tr.ctx, tr.sid, out.ctypes.data)
        assert np.isnan(out).all()
        np.testing.assert_array_equal(tr.get_params(), before)
        tr.close()


def test_an_error_is_reported_once():
    """A call that failed under capture does not fail the next one."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        tr, w = _tracer("wavefront")
        want = tr.render(OPTS).clone()
        with _lost_capture(stream), pytest.raises(L.IptError):
            tr.get_params()
        assert torch.equal(tr.render(OPTS), want)
        tr.close()

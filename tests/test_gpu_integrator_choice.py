"""A context whose program set no integrator runs passes of few paths on the
megakernel and larger ones on the wavefront (28 warps of paths an SM for the
residual pass, 14 for the derivative pass); one that set it runs what it set.
The paths are the same: images are equal bit for bit, and gradients agree to
the rounding of FP32 sums in another order (rel 1e-5)."""
import numpy as np
import pytest
import torch

from paper_1903_07145_gb300 import scenes
from paper_1903_07145_gb300.batch import SceneSet
from paper_1903_07145_gb300.tracer import AdamOptions, TraceOptions, Tracer

pytestmark = pytest.mark.gpu
FLAG_TIMING = 1


def _room():
    return scenes.indoor_room(9, n_cuboids=4, cuboid_sub=2, room_sub=2, n_lights=2, n_views=2, width=40, height=31)


def _runs(tr):
    return {k for k, v in tr.kernel_times(reset=True).items() if v[1]}


def _sizes():
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152
    # (pixels, spp_r, spp_d, residual pass on the megakernel, derivative pass on it)
    return [(1, 1, 1, True, True), (28 * sms, 32, 1, True, True), (28 * sms + 1, 32, 1, False, True),
            (14 * sms, 1, 32, True, True), (14 * sms + 1, 1, 32, True, False)]


@pytest.mark.parametrize("batch,spp_r,spp_d,fwd,adj", _sizes())
def test_passes_choose_by_their_paths(batch, spp_r, spp_d, fwd, adj):
    opts = TraceOptions(spp_r=spp_r, spp_d=spp_d, max_depth=3, pixel_batch=batch)
    got = []
    for chosen in (False, True):
        sc = _room()
        tr = Tracer(sc, seed=4, flags=FLAG_TIMING)
        if chosen:
            tr.configure(integrator="wavefront")
        tr.set_params(sc.gt_params)
        tr.set_targets(np.random.default_rng(2).random((tr.n_pix, 3)).astype(np.float32))
        loss, grad = tr.loss_grad(opts, 5)
        got.append((loss, grad.double().cpu()))
        ran = _runs(tr)
        assert ("forward" in ran) == (fwd and not chosen) and ("wf_shade" in ran) == (not fwd or chosen)
        assert ("adjoint" in ran) == (adj and not chosen) and ("wf_adj_a" in ran) == (not adj or chosen)
        tr.close()
    (la, ga), (lb, gb) = got
    assert abs(la - lb) <= 1e-12 * abs(lb)  # FP64 sums of equal residuals
    assert (ga - gb).norm() <= 1e-5 * gb.norm()


@pytest.mark.parametrize("spp", [1, 7, 8, 9, 33, 64])
def test_a_small_image_is_the_wavefronts(spp):
    imgs = []
    for chosen in (False, True):
        sc = _room()
        tr = Tracer(sc, seed=4, flags=FLAG_TIMING)
        if chosen:
            tr.configure(integrator="wavefront")
        tr.set_params(sc.gt_params)
        imgs.append(tr.render(TraceOptions(spp_r=spp, max_depth=4), view=1, with_msq=True))
        assert ("forward" in _runs(tr)) != chosen
        tr.close()
    assert torch.equal(imgs[0][0], imgs[1][0]) and torch.equal(imgs[0][1], imgs[1][1])


def test_a_batch_recaptures_when_the_program_chooses():
    """The same settings, set by the program: the batch's iterations run the
    wavefront from then on, with the losses of a batch that ran it all along."""
    rows = {}
    for late in (False, True):
        members = [scenes.cornell_variant(k) for k in range(3)]
        ss = SceneSet(members, seed=6)
        if not late:
            ss.configure(integrator="wavefront")
        for i, sc in enumerate(members):
            free = np.zeros((sc.n_segments, 10), np.uint8)
            free[:, 0:3] = 1
            ss.set_params(i, sc.gt_params, free)
            ss.set_targets(i, torch.from_numpy(np.random.default_rng(i).random((ss.n_pix[i], 3))))
        ss.make_batch()
        opts = TraceOptions(spp_r=16, spp_d=2, max_depth=3, pixel_batch=33)
        out = []
        for it in range(4):
            if late and it == 2:
                ss.configure(integrator="wavefront")
            out.append(ss.batch_step(opts, AdamOptions()))
        rows[late] = np.stack(out)
    np.testing.assert_allclose(rows[True], rows[False], rtol=1e-4)


def test_a_pixel_of_more_samples_than_slots_keeps_its_sums():
    """A wavefront too small for one pixel's samples leaves the pass to the
    megakernel, which adds them as a megakernel configured by the program."""
    imgs = []
    for integrator in ("wavefront", "megakernel"):
        sc = _room()
        tr = Tracer(sc, seed=4)
        tr.configure(integrator=integrator, wavefront_slots=1024)
        tr.set_params(sc.gt_params)
        tr.set_targets(np.zeros((tr.n_pix, 3), np.float32))
        small = tr.loss_grad(TraceOptions(spp_r=1030, spp_d=1, max_depth=2, pixel_batch=8), 1)[0]
        imgs.append((tr.render(TraceOptions(spp_r=1030, max_depth=2), view=0), small))
        tr.close()
    assert torch.equal(imgs[0][0], imgs[1][0])
    assert imgs[0][1] == imgs[1][1]

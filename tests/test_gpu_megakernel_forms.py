"""The megakernel's launch forms: one sample a thread with the radiances summed
by a second kernel (up to 2^20 samples) and a pixel's samples in one warp
(more).  Both sum in the same order, so an image is bit-identical whichever
form its launch took; the derivative forms agree to the rounding of their
FP32 sums (rel 1e-5 of the gradient's norm)."""
import numpy as np
import pytest
import torch

from paper_1903_07145_gb300 import scenes
from paper_1903_07145_gb300.tracer import TraceOptions, Tracer

pytestmark = pytest.mark.gpu


def _tracer(views, w, h, seed=4):
    sc = scenes.indoor_room(9, n_cuboids=4, cuboid_sub=2, room_sub=2, n_lights=2, n_views=views, width=w, height=h)
    tr = Tracer(sc, seed=seed)
    tr.configure(integrator="megakernel")
    tr.set_params(sc.gt_params)
    return sc, tr


@pytest.mark.parametrize("spp", [33, 64])
def test_image_does_not_depend_on_the_launch_form(spp):
    # a view alone: below 2^20 samples; all views: above
    sc, tr = _tracer(5, 80, 81)
    opts = TraceOptions(spp_r=spp, max_depth=2)
    n = 80 * 81
    assert n * spp < 1 << 20 < 5 * n * spp
    whole, msq = tr.render(opts, with_msq=True)
    for v in range(5):
        img, m2 = tr.render(opts, view=v, with_msq=True)
        assert torch.equal(img, whole[v * n:(v + 1) * n])
        assert torch.equal(m2, msq[v * n:(v + 1) * n])
    tr.close()


@pytest.mark.parametrize("batch,spp_r,spp_d", [(1, 1, 1), (1, 128, 1), (8, 33, 3), (64, 19, 19), (1217, 1, 1),
                                               (1216, 32, 32), (1217, 32, 32)])
def test_pixel_batches_equal_the_wavefront(batch, spp_r, spp_d):
    sc, tr = _tracer(2, 40, 31)
    rng = np.random.default_rng(2)
    tr.set_targets(rng.random((tr.n_pix, 3)).astype(np.float32))
    opts = TraceOptions(spp_r=spp_r, spp_d=spp_d, max_depth=3, pixel_batch=batch)
    got = []
    for integrator in ("megakernel", "wavefront"):
        tr.configure(integrator=integrator)
        loss, grad = tr.loss_grad(opts, 5)
        got.append((loss, grad.double().cpu()))
    (la, ga), (lb, gb) = got
    assert abs(la - lb) <= 1e-5 * abs(lb)
    assert (ga - gb).norm() <= 1e-5 * gb.norm()
    tr.close()

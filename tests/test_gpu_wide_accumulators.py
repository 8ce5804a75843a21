"""Gradients accumulated in global memory (more segments than shared memory
holds): padded rows and vector reductions against the megakernel's scalar
additions over the same paths.  Both add the same FP32 terms in another
order, at most 1e5 to a row, so they differ by the rounding of such sums: 1e-4
of the gradient's norm bounds it with a wide margin."""
import numpy as np
import pytest
import torch

from paper_1903_07145_gb300 import scenes
from paper_1903_07145_gb300.tracer import TraceOptions, Tracer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", ["lambert_ggx", "disney"])
@pytest.mark.parametrize("spp", [1, 7, 32])
def test_wide_rows_equal_scalar_additions(model, spp):
    room = scenes.indoor_room(21, n_cuboids=14, cuboid_sub=6, room_sub=4, n_lights=1, n_views=1, width=33, height=27)
    sc = scenes.per_triangle(room)
    assert sc.n_segments > 5120
    tr = Tracer(sc, seed=5)
    rng = np.random.default_rng(1)
    tr.set_targets(rng.random((tr.n_pix, 3)).astype(np.float32))
    if model == "disney":
        tr.disney_set_params(scenes.disney_materials(sc, 2))
        call = tr.disney_loss_grad
    else:
        tr.set_params(np.asarray(sc.gt_params) * rng.uniform(0.8, 1.2, (sc.n_segments, 10)))
        call = tr.loss_grad
    opts = TraceOptions(spp_r=spp, spp_d=spp, max_depth=3)
    grads = []
    for integrator in ("megakernel", "wavefront"):
        tr.configure(integrator=integrator)
        grads.append(call(opts, 3)[1].double().cpu())
    assert grads[0].norm() > 0
    for cols in (slice(0, grads[0].shape[1] - 3), slice(grads[0].shape[1] - 3, None)):
        a, b = grads[0][:, cols], grads[1][:, cols]
        assert (a - b).norm() <= 1e-4 * a.norm()
    tr.close()

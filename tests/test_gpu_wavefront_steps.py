"""Steps and shards of images this small on the wavefront too: a program that
sets no integrator runs them on the megakernel (tests/test_gpu_parallel.py)."""
import numpy as np
import pytest
import torch

from paper_1903_07145_gb300 import scenes
from paper_1903_07145_gb300.tracer import AdamOptions, TraceOptions, Tracer

pytestmark = pytest.mark.gpu
OPTS = TraceOptions(spp_r=8, spp_d=8, max_depth=3)


def _tracer(integrator):
    sc = scenes.cornell_box(1000, 32, 32)
    tr = Tracer(sc, seed=5)
    if integrator != "unset":
        tr.configure(integrator)
    tr.set_params(sc.gt_params)
    tr.set_targets(tr.render(OPTS, set_id=2, spp=64))
    tr.set_params(scenes.initial_params(sc, 0.5))
    return tr


@pytest.mark.parametrize("integrator", ["unset", "wavefront", "megakernel"])
def test_shards_sum_to_the_whole(integrator):
    """Uneven shards: FP64 sums of equal residuals, gradients to the rounding
    of FP32 sums in another order."""
    tr = _tracer(integrator)
    loss, grad = tr.loss_grad(OPTS, 3)
    cuts = [0, 1, 130, 131, 700, tr.n_pix]
    parts = [tr.loss_grad_shard(OPTS, 3, a, b - a, tr.n_pix) for a, b in zip(cuts, cuts[1:])]
    assert abs(sum(p[0] for p in parts) - loss) <= 1e-12 * loss
    total = sum(p[1].double() for p in parts)
    assert (total - grad.double()).norm() <= 1e-5 * grad.double().norm()
    tr.close()


def test_steps_agree_between_integrators():
    """Three steps: the losses of parameters that differ only where Adam
    normalised a gradient at the noise of the FP32 sums (as between a shard's
    step and a whole one)."""
    adam = AdamOptions(lr=1e-2)
    got = {}
    for integrator in ("unset", "wavefront", "megakernel"):
        tr = _tracer(integrator)
        got[integrator] = [tr.step(OPTS, adam) for _ in range(3)], tr.get_params()
        tr.close()
    l0, p0 = got["wavefront"]
    for integrator in ("unset", "megakernel"):
        l1, p1 = got[integrator]
        assert abs(l0[0] - l1[0]) <= 1e-5 * abs(l0[0]) and np.allclose(l0, l1, rtol=1e-4, atol=0)
        d = np.abs(p0 - p1)
        assert np.mean(d < 1e-5) >= 0.95 and d.max() <= 6 * adam.lr

"""Single-scene calls between a batch's steps use the scene's own parameters,
and the batch's steps its own, in any order."""
import numpy as np
import pytest
import torch

from paper_1903_07145_gb300 import scenes
from paper_1903_07145_gb300.batch import SceneSet
from paper_1903_07145_gb300.tracer import AdamOptions, TraceOptions

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("integrator", ["unset", "wavefront", "megakernel"])
def test_calls_between_batch_steps_keep_their_parameters(integrator):
    members = [scenes.cornell_variant(k) for k in range(2)]
    opts = TraceOptions(spp_r=8, spp_d=2, max_depth=3)
    losses, images = [], []
    for between in (False, True):
        ss = SceneSet(members, seed=6)
        if integrator != "unset":
            ss.configure(integrator)
        for i, sc in enumerate(members):
            ss.set_params(i, sc.gt_params)
            ss.set_targets(i, torch.from_numpy(np.random.default_rng(i).random((ss.n_pix[i], 3))))
        ss.make_batch()
        rows = []
        for _ in range(3):
            if between:
                images.append([ss.render(i, opts).clone() for i in range(2)])
            rows.append(ss.batch_step(opts, AdamOptions(lr=0.05)))
        losses.append(np.stack(rows))
        ss.close()
    # the steps' gradients are FP32 sums in a varying order
    np.testing.assert_allclose(losses[1], losses[0], rtol=1e-4)
    for later in images[1:]:
        for a, b in zip(later, images[0]):
            assert torch.equal(a, b)

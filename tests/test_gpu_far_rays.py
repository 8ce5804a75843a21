"""Rays whose plane distances overflow (origins at infinity, no direction and
an origin far away) miss, without an error and without a word in the results
of the rays around them."""
import numpy as np
import pytest
import torch

from paper_1903_07145_gb300 import scenes
from paper_1903_07145_gb300.tracer import Tracer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [300, 200003])
def test_overflowing_rays_miss(n):
    sc = scenes.indoor_room(3, n_cuboids=6, cuboid_sub=4, room_sub=4, n_lights=2, n_views=1, width=8, height=8)
    tr = Tracer(sc, seed=1)
    o, d = scenes.random_rays(sc, n, 4)
    want = [v.cpu() for v in tr.trace_rays(torch.from_numpy(o), torch.from_numpy(d))]
    rng = np.random.default_rng(7)
    far = rng.random(n) < 0.3
    kind = rng.integers(0, 3, n)
    sign = rng.choice([-1.0, 1.0], (n, 3)).astype(np.float32)
    o, d = o.copy(), d.copy()
    everywhere = far & (kind == 0)
    o[everywhere] = np.inf * sign[everywhere]
    one_axis = far & (kind == 1)
    o[one_axis, 0] = np.inf * sign[one_axis, 0]
    still = far & (kind == 2)  # a zero component counts as +0: planes behind the origin
    o[still], d[still] = 1e30, 0.0
    got = [v.cpu() for v in tr.trace_rays(torch.from_numpy(o), torch.from_numpy(d))]
    tr.synchronize()
    assert (got[0][far] == -1).all() and torch.isinf(got[1][far]).all()
    for a, b in zip(got, want):
        assert torch.equal(a[~far], b[~far])
    tr.close()

"""ipt_cache_eval and ipt_cache_grad on the caller's arrays: odd row counts,
arrays at every 4-byte alignment, and outputs that share memory with inputs
give the rows that separate, aligned arrays give."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_1903_07145_gb300 import _lib as L
from paper_1903_07145_gb300 import scenes
from paper_1903_07145_gb300.tracer import CacheOptions, Tracer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tracer():
    tr = Tracer(scenes.cornell_box(1000), seed=1)
    tr.configure_cache(CacheOptions())
    rng = np.random.default_rng(3)
    shapes = ((80, 64), (64, 64), (64, 64), (64, 64), (64, 16))
    w = np.concatenate([rng.uniform(-1, 1, s).ravel() * np.sqrt(6.0 / s[0]) for s in shapes])
    tr.set_cache_weights(w, rng.random(L.IPT_CACHE_TABLE_FLOATS, dtype=np.float32) - 0.5)
    yield tr
    tr.close()


def _rows(n, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda k: torch.rand((n, k), device="cuda", generator=g)  # noqa: E731
    unit = lambda v: v / v.norm(dim=1, keepdim=True)  # noqa: E731
    return r(3), unit(r(3) - 0.5), unit(r(3) - 0.5), r(7), r(3)


def _ptr(t):
    return C.c_void_p(t.data_ptr())


def _shifted(t, k):
    """A copy of t whose storage starts k floats past an aligned address."""
    buf = torch.zeros(t.numel() + 8, device="cuda")
    v = buf[k:k + t.numel()].view(t.shape)
    v.copy_(t)
    return v


@pytest.mark.parametrize("n", [1, 15, 127, 129, 1000])
@pytest.mark.parametrize("shift", [1, 3])
def test_eval_at_any_alignment_and_in_place(tracer, n, shift):
    x, d, nn, p7, up = _rows(n)
    rgb, dp = tracer.cache_eval(x, d, nn, p7, upstream=up)
    plain = tracer.cache_eval(x, d, nn, p7)
    assert (rgb - plain).norm() <= 2e-2 * plain.norm()  # FP16 against FP32 table
    args = [_shifted(t, shift) for t in (x, d, nn, p7, up)]
    out, dout = _shifted(torch.zeros(n, 3, device="cuda"), shift), _shifted(torch.zeros(n, 7, device="cuda"), shift)
    L.ipt_cache_eval(tracer.ctx, tracer.sid, n, *[_ptr(t) for t in args], _ptr(out), _ptr(dout))
    tracer.synchronize()
    assert torch.equal(out, rgb) and torch.equal(dout, dp)
    # the prediction over the upstream, the derivative over the parameters
    L.ipt_cache_eval(tracer.ctx, tracer.sid, n, *[_ptr(t) for t in args], _ptr(args[4]), _ptr(args[3]))
    tracer.synchronize()
    assert torch.equal(args[4], rgb) and torch.equal(args[3], dp)
    # the prediction one row further along the positions' array
    big = torch.zeros(n + 1, 3, device="cuda")
    big[:n] = x
    L.ipt_cache_eval(tracer.ctx, tracer.sid, n, _ptr(big), _ptr(d), _ptr(nn), _ptr(p7), None, _ptr(big[1:]), None)
    tracer.synchronize()
    assert torch.equal(big[1:], plain)


@pytest.mark.parametrize("n", [1, 64, 65, 9729, 20000])
def test_grad_at_any_alignment_and_without_outputs(tracer, n):
    x, d, nn, p7, y = _rows(n, 5)
    loss, gw, gt = tracer.cache_grad(x, d, nn, p7, y)
    assert gw.norm() > 0 and gt.norm() > 0
    for shift in (1, 2):
        w2 = _shifted(torch.full_like(gw, 7.0), shift)
        t2 = _shifted(torch.full_like(gt, 7.0), shift)
        l2 = L.ipt_cache_grad(tracer.ctx, tracer.sid, n, _ptr(x), _ptr(d), _ptr(nn), _ptr(p7), _ptr(y), _ptr(w2),
                              _ptr(t2))
        # other order of the same FP32 sums
        assert abs(l2 - loss) <= 1e-9 * loss
        assert (w2 - gw).norm() <= 1e-5 * gw.norm() and (t2 - gt).norm() <= 1e-5 * gt.norm()
    l3, w3, none = tracer.cache_grad(x, d, nn, p7, y, table=False)
    assert none is None and abs(l3 - loss) <= 1e-9 * loss and (w3 - gw).norm() <= 1e-5 * gw.norm()

"""Fused network kernels at the edges of their tiles against the FP64 reference.

Tolerances: the gradient and forward checks compare FP32 sums over 256 neurons and n samples of
values of order one with FP64; 256 * 2^-24 = 1.5e-5 bounds the forward sum's relative rounding
and 1e-3 is the gradient tolerance of the other gradient tests.  The inference numerics round h1
to BF16, reproduced in the reference; a value next to a rounding boundary may fall to the other
side (2^-9 of one of 256 terms), so single results are allowed 1e-3 of the largest.
"""
import numpy as np
import pytest

import paper_1605_02611_gb300 as G
from oracle import mlp as omlp

from gpu_util import require_gpu
from test_gpu_mlp import _bf16, _features, _params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 152 * 128 + 1])
def test_forward_tiles(n):
    require_gpu()
    net = G.Mlp(seed=1)
    th = _params(21)
    net.set_params(th)
    F = _features(22, n)
    ref, _ = omlp.forward(th, F.astype(np.float64))
    g = net.forward(F, inference=False)
    assert np.max(np.abs(g - ref)) < 1.5e-5 * max(1.0, np.max(np.abs(ref)))
    p = omlp.unflatten(th)
    h1 = _bf16(omlp.gelu(F.astype(np.float64) @ p["W1"].T + p["b1"]))
    want = omlp.gelu(h1 @ p["W2"].T + p["b2"]) @ p["W3"] + p["b3"][0]
    got = net.forward(F, inference=True)
    assert np.max(np.abs(got - want)) < 1e-3 * max(1.0, np.max(np.abs(want)))
    net.close()


@pytest.mark.parametrize("n", [2, 63, 65, 152 * 32 + 5])
def test_gradient_tiles(n):
    require_gpu()
    net = G.Mlp(seed=2)
    th = _params(23)
    net.set_params(th)
    F = _features(24, n)
    rng = np.random.default_rng(25)
    P, T = rng.normal(size=n).astype(np.float32), rng.normal(size=n).astype(np.float32)
    Lr, gr = omlp.loss_grad(th, F.astype(np.float64), P.astype(np.float64), T.astype(np.float64))
    for _ in range(2):  # the second call starts from the first one's buffers
        L, g = net.loss_grad(F, P, T)
        assert L == pytest.approx(Lr, rel=1e-5)
        gp, rp = omlp.unflatten(g.astype(np.float64)), omlp.unflatten(gr)
        for name in gp:
            assert np.max(np.abs(gp[name] - rp[name])) < 1e-3 * max(np.max(np.abs(rp[name])), 1e-30), name
    net.close()

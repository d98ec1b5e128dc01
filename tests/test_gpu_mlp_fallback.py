"""A network whose output overflows in the middle of a Davidson solve: the step goes on with the
diagonal correction."""
import numpy as np
import pytest

import paper_1605_02611_gb300 as G
from paper_1605_02611_gb300 import synth

from gpu_util import context_with_mps, require_gpu

pytestmark = pytest.mark.gpu


def test_overflowing_network_gives_the_diagonal_correction():
    """The FP64 path adds in a fixed order, so energy and vector are those of a step without a
    network to the bit."""
    require_gpu()
    K, M, k = 8, 60, 3
    h, eri = synth.integrals(K, 51)
    bonds, T = synth.random_isometric_mps(K, K, 0, M, 52, k)
    net = G.Mlp(seed=4)
    p = net.get_params()
    p[-257:-1] = 3e38  # W3: finite, and its sum over the hidden layer is not
    net.set_params(p)
    assert np.any(~np.isfinite(net.forward(np.ones((4, 5), np.float32), inference=True)))
    out = []
    for mlp in (None, net):
        ctx = context_with_mps(h, eri, K, 0, bonds, T)
        ctx.prepare(k)
        ctx.set_preconditioner(mlp)
        e, _, it, psi = ctx.step(k, 0, M, 1e-9, 30, want_psi=True)
        out.append((e, it, psi))
        cnt = ctx.precond_counters()
        ctx.close()
    assert cnt["fallbacks"] > 0 and cnt["learned"] == 0
    assert out[0][0] == out[1][0] and out[0][1] == out[1][1]
    assert np.array_equal(out[0][2], out[1][2])
    net.close()

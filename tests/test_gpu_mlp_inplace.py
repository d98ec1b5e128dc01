"""The network's output written over its own features."""
import ctypes

import numpy as np
import pytest

import paper_1605_02611_gb300 as G

from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("inference", [0, 1])
@pytest.mark.parametrize("n,at", [(300000, 0), (300000, 900001), (300000, 5 * 300000 - 1), (1, 0)])
def test_output_over_the_features(n, at, inference):
    """A thread block's output lies where another one's features are; every sample is computed by
    itself, so the values are the same to the bit."""
    torch = require_gpu()
    rng = np.random.default_rng(61)
    net = G.Mlp(seed=6)
    net.set_params(rng.normal(0, 0.1, net.nparams).astype(np.float32))
    F = rng.normal(size=(n, 5)).astype(np.float32)
    want = net.forward(F, inference=bool(inference))
    buf = torch.zeros(6 * n, device="cuda")
    buf[:5 * n] = torch.tensor(F.reshape(-1))
    torch.cuda.synchronize()
    net._check(net.lib.gbdmrg_mlp_forward(net.h, ctypes.c_void_p(buf.data_ptr()), n,
                                          ctypes.c_void_p(buf.data_ptr() + 4 * at), inference, 1), "forward")
    assert np.array_equal(buf[at:at + n].cpu().numpy(), want)
    net.close()

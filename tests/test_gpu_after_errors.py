"""What a call leaves behind when a device allocation fails: an error status, and objects that work."""
import numpy as np
import pytest

import paper_1605_02611_gb300 as G
from paper_1605_02611_gb300 import synth

from gpu_util import context_with_mps, require_gpu

pytestmark = pytest.mark.gpu


def _context(precision=0, K=6, M=30, k=2):
    h, eri = synth.integrals(K, 41)
    bonds, T = synth.random_isometric_mps(K, K, 0, M, 42, k)
    ctx = context_with_mps(h, eri, K, 0, bonds, T)
    ctx.set_precision(precision)
    ctx.prepare(k)
    return ctx


def test_an_error_is_reported_once():
    """The launch check of the next call does not report the failed allocation again."""
    require_gpu()
    ctx = _context(5)
    x = np.random.default_rng(43).normal(size=ctx.nnz)
    ref, _ = ctx.sigma(x)
    with pytest.raises(G.GbdmrgError, match="ENOMEM"):
        ctx.set_harvest(1 << 40, 1, 0)  # 22 TB
    got, _ = ctx.sigma(x)
    assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max()
    ctx.close()

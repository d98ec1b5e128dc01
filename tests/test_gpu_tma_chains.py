"""Two- and three-slice sigma with long contraction blocks: terms of more pieces than the
straight-line code takes, than two CTAs' rings hold, and than any ring holds (slice pair by slice
pair), against the FP64 path.  Bars as for the other sliced sigmas: operands to ~2^-16 or better,
FP32 accumulation ~1e-5, so 1e-4 in norm and 2e-4 of the largest element."""
import numpy as np
import pytest

from paper_1605_02611_gb300 import synth

from gpu_util import context_with_mps, rel_err, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [5, 6])
@pytest.mark.parametrize("K,M,spread,longest", [
    (12, 1000, 1.0, 100),  # 7 pieces
    (14, 800, 2.0, 266),   # 17 pieces
])
def test_long_terms(K, M, spread, longest, precision):
    require_gpu()
    k = K // 2 - 1
    h, eri = synth.integrals(K, 900 + K)
    bonds, T = synth.random_isometric_mps(K, K, 0, M, 901, k, spread)
    assert max(bonds[k].dim) == longest
    ctx = context_with_mps(h, eri, K, 0, bonds, T)
    ctx.set_env_precision(3)
    ctx.prepare(k)
    x = np.random.default_rng(902).normal(size=ctx.nnz)
    y64, _ = ctx.sigma(x)
    ctx.set_precision(precision)
    ctx.prepare(k)
    y, _ = ctx.sigma(x)
    assert np.linalg.norm(y - y64) / np.linalg.norm(y64) < 1e-4
    assert rel_err(y, y64) < 2e-4
    y2, _ = ctx.sigma(x)
    assert np.linalg.norm(y2 - y) <= 1e-5 * np.linalg.norm(y)
    ctx.close()

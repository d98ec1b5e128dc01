"""Contraction blocks longer than a term may be on the two- and three-slice sigma are cut into several
terms, alone and in a batch.

Sectors of 96, 97, 112 and 113 states are 6 pieces (a whole term in two slices), 7 (two parts) and 8;
266 states are 17 pieces.  Bars as for the other sliced sigmas: operands to ~2^-16 or better, FP32
accumulation ~1e-5, so 1e-4 in norm and 2e-4 of the largest element.
"""
import numpy as np
import pytest

import paper_1605_02611_gb300 as G
from paper_1605_02611_gb300 import synth

from gpu_util import context_with_mps, rel_err, require_gpu

pytestmark = pytest.mark.gpu


def _problem(K, M, spread, precision, seed, keep=False):
    k = K // 2 - 1
    h, eri = synth.integrals(K, seed)
    bonds, T = synth.random_isometric_mps(K, K, 0, M, seed + 1, k, spread)
    ctx = context_with_mps(h, eri, K, 0, bonds, T)
    ctx.set_env_precision(3)
    ctx.keep_host_plans(keep)
    ctx.set_precision(precision)
    ctx.prepare(k)
    return ctx, k, max(bonds[k].dim)


@pytest.mark.parametrize("precision", [5, 6])
@pytest.mark.parametrize("K,M,spread,longest", [
    (14, 537, 1.0, 96), (14, 542, 1.0, 97), (14, 633, 1.0, 112), (14, 638, 1.0, 113)])
def test_cut_terms(K, M, spread, longest, precision):
    require_gpu()
    ctx, k, top = _problem(K, M, spread, 0, 950)
    assert top == longest
    x = np.random.default_rng(951).normal(size=ctx.nnz)
    y64, _ = ctx.sigma(x)
    ctx.set_precision(precision)
    ctx.plan(k)
    y, _ = ctx.sigma(x)
    assert np.linalg.norm(y - y64) / np.linalg.norm(y64) < 1e-4
    assert rel_err(y, y64) < 2e-4
    ctx.close()


@pytest.mark.parametrize("precision", [5, 6])
def test_long_blocks_run_at_the_rate_of_short_ones(precision):
    """Multiply-adds per second with sectors of up to 266 states and with those of up to 83: a block
    is cheaper per multiply-add the longer it is."""
    torch = require_gpu()

    def rate(K, M, spread):
        ctx, _, _ = _problem(K, M, spread, precision, 960)
        x = torch.tensor(np.random.default_rng(961).normal(size=ctx.nnz), device="cuda")
        y = torch.empty_like(x)
        torch.cuda.synchronize()
        flops = ctx.sigma_device(x.data_ptr(), y.data_ptr())
        ms = min(ctx.sigma_timing(3, x.data_ptr(), y.data_ptr()) for _ in range(3))
        ctx.close()
        return flops / ms

    assert rate(14, 800, 2.0) > rate(20, 800, 1.0)


def test_batch_of_short_and_long_blocks():
    """Problems whose rings do not fit each other: narrow ones beside ones that fill a ring, in one
    batch.  As one by one but for the order of the FP32 additions of the split stage-2 tiles (at most
    about 100 per element, 6e-8 each, in random directions)."""
    torch = require_gpu()
    ctxs, xs, ys, ref = [], [], [], []
    for i, (K, M, spread, p) in enumerate([(8, 60, 1.0, 2), (14, 800, 2.0, 2), (12, 700, 1.0, 3), (12, 900, 1.0, 2),
                                           (14, 800, 2.0, 3), (10, 200, 1.0, 2), (14, 542, 1.0, 2)]):
        ctx, _, _ = _problem(K, M, spread, p, 970 + 10 * i, keep=True)
        x = np.random.default_rng(980 + i).normal(size=ctx.nnz)
        ref.append(ctx.sigma(x)[0])
        ctxs.append(ctx)
        xs.append(torch.tensor(x, device="cuda"))
        ys.append(torch.zeros_like(xs[-1]))
    torch.cuda.synchronize()
    b = G.Batch(ctxs)
    for use_graph in (False, True, True):
        for y in ys:
            y.zero_()
        torch.cuda.synchronize()
        b.sigma([x.data_ptr() for x in xs], [y.data_ptr() for y in ys], use_graph)
        for y, r in zip(ys, ref):
            assert np.linalg.norm(y.cpu().numpy() - r) <= 1e-6 * np.linalg.norm(r)
    b.close()

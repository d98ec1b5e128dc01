"""One batch over problems of different slice counts and numbers of chunks: the work lists
of each slice count go into a launch of their own, chunk by chunk."""
import numpy as np
import pytest

import paper_1605_02611_gb300 as G
from paper_1605_02611_gb300 import synth

from gpu_util import context_with_mps, require_gpu

pytestmark = pytest.mark.gpu

# (K, M, k, precision, chunk budget in MB)
PROBLEMS = [(6, 20, 2, 3, 2048), (10, 600, 3, 2, 1), (8, 100, 3, 1, 2048), (10, 600, 4, 2, 2048), (6, 4, 0, 1, 1)]


@pytest.mark.parametrize("order", [[0, 1, 2, 3, 4], [4, 2, 3, 0, 1], [2]])
def test_batch_of_mixed_slices_and_chunks(order):
    torch = require_gpu()
    ctxs, xs, ys, ref = [], [], [], []
    for i in order:
        K, M, k, precision, mb = PROBLEMS[i]
        h, eri = synth.integrals(K, 400 + i)
        bonds, T = synth.random_isometric_mps(K, K, 0, M, 410 + i, k, 0.5)
        ctx = context_with_mps(h, eri, K, 0, bonds, T)
        ctx.set_precision(precision)
        ctx.set_chunk_budget(mb)
        ctx.keep_host_plans(True)
        ctx.prepare(k)
        x = ctx.pack(synth.random_psi(bonds[k], bonds[k + 2], 420 + i))
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
            # the same tiles and products as one by one; the FP32 additions of the split stage-2
            # tiles (at most about 100 per element, 6e-8 each, in random directions) may change order
            assert np.linalg.norm(y.cpu().numpy() - r) <= 1e-6 * np.linalg.norm(r)
    b.close()

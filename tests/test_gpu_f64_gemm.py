"""FP64 grouped GEMM: every tile edge and lane mapping against the oracle's sigma and diagonal.

The tolerance is that of the FP64 path against the oracle (relative 1e-11 of the largest
element): the kernel adds the same products in FP64, only the grouping of a sum may differ.
"""
import numpy as np
import pytest

from oracle import mps as omps
from paper_1605_02611_gb300 import synth

from gpu_util import context_with_mps, rel_err, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,two_sz,M,k", [
    (4, 4, 0, 1, 1),       # single-element blocks: many lanes share one output
    (5, 4, 0, 7, 1),       # blocks of a few elements
    (6, 6, 0, 64, 0),      # one-row blocks at the left edge, long term lists
    (6, 6, 0, 64, 4),      # and at the right edge
    (8, 8, 0, 40, 2),      # ragged blocks below the smallest tile edge
    (8, 7, 1, 256, 3),     # full bonds, odd particle number: edges of 8 and 16
    (9, 9, 1, 400, 3),     # blocks larger than the smallest edge chosen
])
def test_sigma_and_env_against_oracle(K, N, two_sz, M, k):
    require_gpu()
    h, eri = synth.integrals(K, 40 + K)
    bonds, T = synth.random_mps(K, N, two_sz, M, 41 + M)
    Na, Nb = (N + two_sz) // 2, (N - two_sz) // 2
    psi = synth.random_psi(bonds[k], bonds[k + 2], 42)
    ref = omps.sigma(T, k, psi, h, eri, Na, Nb)
    ctx = context_with_mps(h, eri, N, two_sz, bonds, T)
    ctx.prepare(k)  # the environments come from the same kernel (transposed operands)
    sig, _ = ctx.sigma(ctx.pack(psi))
    assert rel_err(sig, ctx.pack(ref)) < 1e-11
    # the diagonal is the quadratic form of unit vectors
    d = ctx.diag()
    for i in {0, ctx.nnz // 2, ctx.nnz - 1}:
        e = np.zeros(ctx.nnz)
        e[i] = 1.0
        assert abs(ctx.sigma(e)[0][i] - d[i]) < 1e-11 * np.abs(d).max()

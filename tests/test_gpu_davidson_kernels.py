"""Small eigenproblems and reductions of the Davidson solve and the decimation, through the calls
that use them.

A step with a bond dimension of at least the full space keeps the whole wavefunction, so the
product of the two new site tensors is psi up to the rounding of the sector eigenvectors (the
eigenvalues and vectors of d <= 32 sectors come from the Jacobi kernel, larger ones from the library
solver): 1e-10 leaves room for d * 2^-52 and the truncation of weights below 1e-14.
"""
import numpy as np
import pytest

from paper_1605_02611_gb300 import synth

from gpu_util import context_with_mps, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,two_sz,M,direction", [
    (4, 4, 0, 16, 0),      # sectors of 1 to 4 rows
    (5, 5, 1, 16, 1),      # odd dimensions: a rotation pair with a dummy index
    (7, 7, 1, 64, 0),      # up to 36 rows: both solvers in one decimation
    (8, 8, 0, 256, 1),
])
def test_step_keeps_psi(K, N, two_sz, M, direction):
    require_gpu()
    h, eri = synth.integrals(K, 60 + K)
    k = K // 2 - 1
    bonds, T = synth.random_isometric_mps(K, N, two_sz, M, 61, k)
    ctx = context_with_mps(h, eri, N, two_sz, bonds, T)
    ctx.prepare(k)
    nl, nr = bonds[k].total, bonds[k + 2].total
    _, dw, _, psi = ctx.step(k, direction, 4 * M, 1e-9, 12, want_psi=True)
    A, B = ctx.get_mps(k), ctx.get_mps(k + 1)
    full = np.einsum("anb,bmc->anmc", A, B)
    assert np.linalg.norm(full - ctx.unpack(psi, (nl, 4, 4, nr))) < 1e-10
    assert dw < 1e-12
    # the kept vectors are orthonormal
    Q = A.reshape(-1, A.shape[2]).T if direction == 0 else B.reshape(B.shape[0], -1)
    assert np.abs(Q @ Q.T - np.eye(len(Q))).max() < 1e-12


@pytest.mark.parametrize("max_iter", [1, 2, 23, 24, 40])
def test_ritz_value_is_variational_and_converges(max_iter):
    """The Ritz value of m = 1, 2, ... subspace vectors (restart after 24) never rises and, at 40
    iterations, has reached the dense lowest eigenvalue of H_eff."""
    require_gpu()
    K, N, M, k = 5, 4, 9, 1
    h, eri = synth.integrals(K, 71)
    bonds, T = synth.random_isometric_mps(K, N, 0, M, 72, k)
    ctx = context_with_mps(h, eri, N, 0, bonds, T)
    ctx.prepare(k)
    n = ctx.nnz
    H = np.stack([ctx.sigma(e)[0] for e in np.eye(n)])
    w = np.linalg.eigvalsh(0.5 * (H + H.T))
    x = np.random.default_rng(73).normal(size=n)
    e, _, _, _ = ctx.step(k, 0, 64, 1e-10, max_iter, psi_in=x)
    assert e > w[0] - 1e-10 * abs(w[0])
    if max_iter == 40:
        assert abs(e - w[0]) < 1e-9 * abs(w[0])
    if max_iter == 1:
        assert abs(e - x @ H @ x / (x @ x)) < 1e-10 * abs(w).max()

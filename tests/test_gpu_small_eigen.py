"""The Jacobi eigensolvers of the decimation's small sectors and of the Rayleigh-Ritz step, alone.

Every element of a matrix of n rows is turned some 10 n times until it converges, each time with a
rounding of 2^-53 of the norm, in random directions: 10 n 2^-52 |A| bounds residuals and values (1e-13
|A| at n = 48).
"""
import numpy as np
import pytest

import paper_1605_02611_gb300 as G
from paper_1605_02611_gb300 import synth

from gpu_util import context_with_mps, require_gpu

pytestmark = pytest.mark.gpu


def _spectra(n):
    i = np.arange(n)
    two = np.where(i < 2, -1.0, i / n)
    yield "random", np.random.default_rng(n).normal(size=n)
    yield "lowest twice", two
    for gap in (1e-2, 1e-3, 3e-4, 1e-4, 1e-8, 1e-15):  # about the line below which the Ritz step takes FP64 throughout
        w = two.copy()
        w[0] -= gap
        yield f"gap {gap}", w
    yield "graded", 10.0 ** -i
    yield "two values", np.where(i < n // 2, 0.25, 1.0)
    yield "all alike", np.ones(n)
    yield "zero", np.zeros(n)


def _matrices(n):
    rng = np.random.default_rng(100 + n)
    for name, w in _spectra(n):
        q, _ = np.linalg.qr(rng.normal(size=(n, n)))
        a = (q * w) @ q.T
        yield name, 0.5 * (a + a.T)


@pytest.mark.parametrize("n", [1, 2, 3, 24, 31, 32])
def test_sector_kernel(n):
    require_gpu()
    for name, a in _matrices(n):
        w, V = G.eigen_selftest(0, a)
        tol = 10 * n * 2.0 ** -52 * max(np.linalg.norm(a), 1e-300)
        assert np.abs(w - np.linalg.eigvalsh(a)).max() <= tol, name
        assert np.all(np.diff(w) >= 0), name
        assert np.abs(a @ V.T - V.T * w).max() <= tol, name
        assert np.abs(V @ V.T - np.eye(n)).max() <= 10 * n * 2.0 ** -52, name


@pytest.mark.parametrize("n", [1, 2, 24, 25, 47, 48])
def test_ritz_kernel(n):
    require_gpu()
    for name, a in _matrices(n):
        w, v = G.eigen_selftest(1, a)
        tol = 10 * n * 2.0 ** -52 * max(np.linalg.norm(a), 1e-300)
        assert abs(w[0] - np.linalg.eigvalsh(a)[0]) <= tol, name
        assert np.linalg.norm(a @ v - w[0] * v) <= tol * np.sqrt(n), name
        assert abs(np.linalg.norm(v) - 1) <= 10 * n * 2.0 ** -52, name


@pytest.mark.parametrize("which,n", [(0, 32), (1, 48)])
def test_no_convergence_is_reported(which, n):
    """One sweep does not do, nor does any number of them for a matrix with a NaN or an infinity."""
    require_gpu()
    a = np.random.default_rng(5).normal(size=(n, n))
    a = a + a.T
    with pytest.raises(G.GbdmrgError, match="ENOCONV"):
        G.eigen_selftest(which, a, max_sweeps=1)
    for bad in (np.nan, np.inf):
        b = a.copy()
        b[3, 7] = b[7, 3] = bad
        with pytest.raises(G.GbdmrgError, match="ENOCONV"):
            G.eigen_selftest(which, b)


def test_ritz_value_never_rises():
    """Solves of 1, 2, ... iterations (the subspace restarts after 24 vectors): the FP64 path is the
    same from solve to solve, so the value can rise by its rounding only."""
    require_gpu()
    K, N, M, k = 5, 4, 9, 1
    h, eri = synth.integrals(K, 71)
    bonds, T = synth.random_isometric_mps(K, N, 0, M, 72, k)
    x, e = None, []
    for it in list(range(1, 30)) + [40]:
        ctx = context_with_mps(h, eri, N, 0, bonds, T)
        ctx.prepare(k)
        if x is None:
            x = np.random.default_rng(73).normal(size=ctx.nnz)
        e.append(ctx.step(k, 0, 64, 1e-10, it, psi_in=x)[0])
        ctx.close()
    assert np.diff(e).max() <= 1e-12 * np.abs(e).max()
    assert e[0] - e[-1] > 1e-3 * abs(e[-1])

"""Levels of pencils whose S is ill conditioned.  The blocked factorisation goes through
explicit inverses of the diagonal blocks, each product refined once; without the
refinement the levels' error is three times that of substitutions.

Measure: the mean error over eight pencils against 60-digit arithmetic, relative to
that of NumPy's Cholesky factor and substitutions in FP64.  Emulated in NumPy, the
square-root-free elimination with refined products has 1.9 times their error at
worst and means of eight scatter by 1.3: at most 2.5."""
import numpy as np
import pytest
import scipy.linalg as sl

from gpu_util import gpu_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


def _pencil(n, cond, seed):
    """S = Q D Q^T, H = F diag(E) F^T with F = Q sqrt(D) R: the levels are E, up to the
    rounding of the products (made in extended precision)."""
    r = np.random.default_rng(seed)
    Q = np.linalg.qr(r.standard_normal((n, n)))[0]
    R = np.linalg.qr(r.standard_normal((n, n)))[0]
    s = np.exp(np.linspace(0.0, -np.log(cond), n))
    E = np.sort(r.uniform(-1.0, 5.0, n))
    F = (Q * np.sqrt(s)) @ R
    H, S = (F * E) @ F.T, (Q * s) @ Q.T
    return 0.5 * (H + H.T), 0.5 * (S + S.T)


def _exact(H, S):
    """Levels in 60-digit arithmetic of the matrices as they are."""
    mp = pytest.importorskip("mpmath")
    with mp.workdps(60):
        L = mp.cholesky(mp.matrix(S.tolist()))
        Li = L ** -1
        A = Li * mp.matrix(H.tolist()) * Li.T
        return np.sort(np.array([float(x) for x in mp.eigsy(A, eigvals_only=True)]))


@pytest.mark.parametrize("cond", [1e7, 1e10])
def test_error_against_substitutions(ofm, cond):
    n, got, want = 40, [], []
    for seed in range(8):
        H, S = _pencil(n, cond, seed)
        E = _exact(H, S)
        L = np.linalg.cholesky(S)
        X = sl.solve_triangular(L, H, lower=True)
        A = sl.solve_triangular(L, X.T, lower=True)
        want.append(np.abs(np.linalg.eigvalsh(0.5 * (A + A.T)) - E).max())
        ctx = ofm.Context()
        ctx.set_dense_HS(H, S)
        got.append(np.abs(ctx.eigs_by_index(0, n) - E).max())
    assert np.mean(got) <= 2.5 * np.mean(want), (np.mean(got), np.mean(want))

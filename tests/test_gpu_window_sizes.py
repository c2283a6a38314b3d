"""The window solve at the edges of its blocks: matrix orders around the 32-row
blocks and 16-column strips of the factorisation, the one-CTA reduction's range
and one past it, an H given symmetric only up to rounding, and a pivot that is
not positive in a later block, against LAPACK.

Tolerance of an eigenvalue: the Cholesky route is backward stable up to the
conditioning of S, |dE| <= (8 n + 16) u kappa(S) max |E|."""
import numpy as np
import pytest
import scipy.linalg as sl

from gpu_util import U64, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


def pencil(n, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, n))
    S = X @ X.T / n + 0.3 * np.eye(n)
    H = rng.standard_normal((n, n))
    return 0.5 * (H + H.T), 0.5 * (S + S.T)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 15, 16, 17, 31, 32, 33, 47, 48, 49, 63, 64, 65, 66, 95, 97, 112, 129,
                               160, 321])
def test_eigenvalues_and_vectors_at_block_edges(ofm, n):
    H, S = pencil(n, n)
    skew = np.triu(np.random.default_rng(n + 1).standard_normal((n, n)), 1) * 1e-15
    ctx = ofm.Context()
    ctx.set_dense_HS(H + skew, S)
    E = sl.eigh(H, S, eigvals_only=True)
    tol = (8 * n + 16) * U64 * np.linalg.cond(S) * np.abs(E).max()
    assert np.max(np.abs(ctx.eigs_by_index(0, n) - E)) <= tol
    Eg, C, cnt = ctx.window_eigs(E[0] - 1.0, E[-1] + 1.0, vectors=True, n_basis=n)
    assert cnt == n
    assert np.max(np.abs(Eg - E)) <= tol
    # the residual of a normalised vector against the matrices' norms
    res = np.linalg.norm(H @ C - S @ C * Eg, axis=0)
    assert np.all(res <= 1e3 * n * U64 * np.linalg.cond(S) * np.linalg.norm(C, axis=0) * np.linalg.norm(H, 2))


@pytest.mark.parametrize("n,bad", [(40, 33), (96, 70), (33, 32)])
def test_pivot_of_a_later_block(ofm, n, bad):
    H, S = pencil(n, n)
    S[bad, bad] = -1.0
    ctx = ofm.Context()
    ctx.set_dense_HS(H, S)
    with pytest.raises(ofm.OFMError) as e:
        ctx.eigs_by_index(0, 1)
    assert e.value.status == ofm.OFM_ERR_NOT_POSDEF and f"pivot {bad} " in str(e.value)


@pytest.mark.parametrize("n", [4266, 4267])
def test_vectors_at_the_end_of_the_row_ring(ofm, n):
    # a reflection of known levels; the back-transformation stages its rows up to n = 4266
    D = np.linspace(0.0, 1000.0, n)
    w = np.random.default_rng(n).standard_normal(n)
    w /= np.linalg.norm(w)
    Dw = D * w
    H = -2.0 * (np.outer(w, Dw) + np.outer(Dw, w)) + 4.0 * (w @ Dw) * np.outer(w, w)
    H[np.diag_indices(n)] += D
    ctx = ofm.Context()
    ctx.set_dense_HS(H, np.eye(n))
    E, C, cnt = ctx.window_eigs(-0.1, D[2] + 0.1, max_out=4, vectors=True, n_basis=n)
    assert cnt == 3
    assert np.max(np.abs(E - D[:3])) <= (8 * n + 16) * U64 * 1000.0
    assert np.max(np.linalg.norm(H @ C - C * E, axis=0)) <= 64 * n * U64 * 1000.0

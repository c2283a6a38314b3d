"""The one-CTA tridiagonal reduction (3 <= n <= 64): its warps hand rows over by
named barriers, so the same small pencils, solved again and again, give bitwise
the same levels, and those of LAPACK.

Tolerance as in test_gpu_window_sizes: |dE| <= (8 n + 16) u kappa(S) max |E|."""
import numpy as np
import pytest
import scipy.linalg as sl

from gpu_util import U64, gpu_lib
from test_gpu_window_sizes import pencil

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


@pytest.mark.parametrize("n", [3, 4, 5, 6, 7, 8, 12, 13, 24, 31, 33, 48, 63, 64])
def test_repeated_small_solves_agree_bitwise(ofm, n):
    H, S = pencil(n, 500 + n)
    E = sl.eigh(H, S, eigvals_only=True)
    tol = (8 * n + 16) * U64 * np.linalg.cond(S) * np.abs(E).max()
    ctx = ofm.Context()
    first = None
    for _ in range(60):
        ctx.set_dense_HS(H, S)   # drops the factorisation: every pass reduces anew
        got = np.array(ctx.eigs_by_index(0, n))
        if first is None:
            first = got
            assert np.max(np.abs(got - E)) <= tol
        assert np.array_equal(got, first)

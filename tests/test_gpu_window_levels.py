"""Levels by index where the search for one changes its steps: levels that are
multiple, close (gaps of 1e-12 to 1e-3), of very different sizes, and zero,
for few and many wanted levels, against the matrix's own."""
import numpy as np
import pytest

from gpu_util import U64, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


SPECTRA = {
    "close": np.concatenate([[1.0, 1.0, 1.0], 1 + 10.0 ** np.arange(-12, -2), np.linspace(-2, 3, 40)]),
    "graded": np.concatenate([[0.0], 10.0 ** np.arange(-14.0, 3.0), -(10.0 ** np.arange(-14.0, 3.0))]),
    "pairs": np.repeat(np.linspace(-1, 1, 30), 2),
    "even": np.linspace(-1, 5, 400),
    "one": np.array([0.37]),
}


@pytest.mark.parametrize("name", sorted(SPECTRA))
def test_levels_by_index(ofm, name):
    E = np.sort(SPECTRA[name])
    n = len(E)
    Q = np.linalg.qr(np.random.default_rng(n).standard_normal((n, n)))[0]
    H = (Q * E) @ Q.T
    ctx = ofm.Context()
    ctx.set_dense_HS(0.5 * (H + H.T), np.eye(n))
    tol = (8 * n + 16) * U64 * np.abs(E).max()
    assert np.max(np.abs(ctx.eigs_by_index(0, n) - E)) <= tol
    k = n // 3
    assert np.max(np.abs(ctx.eigs_by_index(k, k + 1) - E[k:k + 1])) <= tol

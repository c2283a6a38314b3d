"""The eigensolver's block operations at the edges of their tiles: box extents
that split into whole and ragged 4 x 2 patches, boxes that span one, two or
three dimensions of the grid, planes too large for the on-chip filter, and
block widths around the register tiles of the Gram, the rotation and the
one-sided Jacobi; energies against the oracle's, residuals of the returned
states recomputed in FP64."""
import numpy as np
import pytest

from ofm_inputs import Fragment, small_workload
from oracle import ofm_oracle as O

from gpu_util import U32, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


def _check(ofm, grid_n, frags, storage, iters=0):
    """iters > 0: that many iterations only, the residuals as they are then."""
    wl = small_workload(grid_n, frags=frags, seed=11)
    H = O.hamiltonian(wl.grid, wl.V)
    ctx = ofm.Context()
    ctx.set_checks(True)      # guard bands of every buffer read after the call
    ctx.build_fragments(wl.grid, wl.V, frags, storage=storage)
    eps, res, _ = ctx.fragment_eigs(max_iter=iters, allow_not_converged=iters > 0)
    u = 0.0 if storage == "fp64" else U32
    top = 12.0 / wl.grid.h ** 2 + np.abs(wl.V).max()     # bound of |H|
    if not iters:
        assert res.max() <= (1e-9 if storage == "fp64" else 1e-5)
    k = 0
    for a, f in enumerate(frags):
        e, r = eps[k:k + f.n_states], res[k:k + f.n_states]
        k += f.n_states
        Hf = O.fragment_hamiltonian(H, wl.grid, f)
        want = np.linalg.eigvalsh(Hf.toarray())
        # an eigenvalue lies within the residual of a Ritz value; in FP32 the
        # values carry a few roundings of |H|
        near = np.min(np.abs(e[:, None] - want[None]), axis=1)
        assert np.all(near <= r + 8 * u * top + 1e-12), (a, f)
        if not iters:
            assert np.max(np.abs(e - want[:f.n_states])) <= r.max() + 8 * u * top + 1e-12, (a, f)
        # the reported residuals are the states' own (stored in FP32: one
        # rounding of |H| on top)
        P = ctx.get_fragment_states(a)
        own = np.linalg.norm(Hf @ P - P * e, axis=0)
        assert np.all(np.abs(own - r) <= 0.02 * r + 6 * u * top + 1e-11), (a, f)
        assert np.max(np.abs(P.T @ P - np.eye(f.n_states))) <= (1e-12 if storage == "fp64" else 64 * u), (a, f)


@pytest.mark.parametrize("storage", ["fp32", "fp64"])
@pytest.mark.parametrize("ext", [(4, 2, 9), (7, 1, 12), (1, 9, 10), (3, 3, 5), (2, 13, 6)])
def test_thin_boxes(ofm, ext, storage):
    n = tuple(e + 3 for e in ext)
    _check(ofm, n, [Fragment((1, 2, 1), ext, 5), Fragment((3, 0, 2), ext, 3)], storage, iters=3)


@pytest.mark.parametrize("storage", ["fp32", "fp64"])
@pytest.mark.parametrize("ext", [(8, 8, 8), (5, 7, 6), (9, 6, 7), (10, 5, 9), (13, 11, 5), (11, 9, 10)])
def test_patch_edges(ofm, ext, storage):
    n = tuple(e + 3 for e in ext)
    P = int(np.prod(ext))
    _check(ofm, n, [Fragment((1, 2, 1), ext, min(5, P - 2)), Fragment((3, 0, 2), ext, min(3, P - 2))], storage)


@pytest.mark.parametrize("storage", ["fp32", "fp64"])
@pytest.mark.parametrize("span", [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (0, 1, 1), (1, 0, 1), (1, 1, 1)])
def test_spanned_dimensions(ofm, span, storage):
    n = (9, 10, 7)
    ext = tuple(n[d] if span[d] else n[d] - 3 for d in range(3))
    _check(ofm, n, [Fragment((2, 1, 3), ext, 4), Fragment((0, 3, 1), (6, 5, 4), 6)], storage)


@pytest.mark.parametrize("ext", [(72, 60, 2), (2, 62, 70)])
def test_plane_too_large_for_the_chip(ofm, ext):
    # no axis order leaves a plane of at most 448 patches with the long axes in it
    n = tuple(e + 3 for e in ext)
    wl = small_workload(n, frags=[Fragment((0, 0, 0), ext, 3)], seed=2)
    ctx = ofm.Context()
    ctx.build_fragments(wl.grid, wl.V, wl.frags, storage="fp32")
    eps, res, _ = ctx.fragment_eigs()
    H = O.hamiltonian(wl.grid, wl.V)
    want, _ = O.fragment_eigs(H, wl.grid, wl.frags[0])
    assert res.max() <= 1e-5
    assert np.max(np.abs(eps - want)) <= 1e-5 + 8 * U32 * (12.0 / wl.grid.h ** 2 + np.abs(wl.V).max())


@pytest.mark.parametrize("storage,states", [("fp32", s) for s in (1, 3, 4, 13, 25, 26, 51, 52, 77, 102, 103, 140)] +
                         [("fp64", s) for s in (1, 2, 12, 13, 25, 26, 60, 90)])
def test_block_widths(ofm, storage, states):
    # blocks of states + max(4, states / 4) vectors
    _check(ofm, (15, 13, 12), [Fragment((1, 1, 1), (11, 9, 8), states), Fragment((2, 3, 0), (8, 8, 6), max(1, states // 3))],
           storage)

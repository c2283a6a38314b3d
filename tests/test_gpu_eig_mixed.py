"""Fragments that the on-chip filter takes beside ones that go one step per
launch (boxes that span the whole grid, planes of more than 3584 points): both
kinds end in the same block whatever the degree's parity, each as if solved alone;
the steps' four-point rows at every remainder and periodic edge; thin boxes laid
out along their longer axes.

FP32 levels within the residual (at most 1e-5) and a few roundings of |H|; the
returned states' own residuals as reported, as in test_gpu_eig_blocks."""
import numpy as np
import pytest

from ofm_inputs import Fragment, small_workload
from oracle import ofm_oracle as O

from gpu_util import U32, gpu_lib
from test_gpu_eig_blocks import _check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


@pytest.mark.parametrize("degree", [1, 2, 6, 7, 8, 31, 32])
def test_spanning_box_beside_others(ofm, degree):
    n = (12, 11, 10)
    frags = [Fragment((0, 0, 0), n, 4), Fragment((3, 2, 1), (7, 6, 5), 3), Fragment((9, 8, 4), (8, 4, 8), 5)]
    wl = small_workload(n, frags=frags, seed=3)
    H = O.hamiltonian(wl.grid, wl.V)
    ctx = ofm.Context()
    ctx.set_checks(True)
    ctx.build_fragments(wl.grid, wl.V, frags, storage="fp32")
    # three passes at these degrees need not converge: the residuals as they are then
    eps, res, _ = ctx.fragment_eigs(degree=degree, max_iter=3, allow_not_converged=True)
    top = 12.0 / wl.grid.h ** 2 + np.abs(wl.V).max()
    k = 0
    for a, f in enumerate(frags):
        e, r = eps[k:k + f.n_states], res[k:k + f.n_states]
        k += f.n_states
        Hf = O.fragment_hamiltonian(H, wl.grid, f)
        want = np.linalg.eigvalsh(Hf.toarray())
        assert np.all(np.min(np.abs(e[:, None] - want[None]), axis=1) <= r + 8 * U32 * top)
        P = ctx.get_fragment_states(a)
        own = np.linalg.norm(Hf @ P - P * e, axis=0)
        assert np.all(np.abs(own - r) <= 0.02 * r + 6 * U32 * top), (a, degree)


@pytest.mark.parametrize("n", [(8, 7, 6), (9, 7, 6), (10, 6, 9), (11, 9, 7), (13, 5, 6)])
def test_spanning_box_converges(ofm, n):
    _check(ofm, n, [Fragment((0, 0, 0), n, 4), Fragment((1, 1, 0), (5, 3, 4), 3)], "fp32")


@pytest.mark.parametrize("ext", [(61, 60, 62), (62, 63, 61), (63, 60, 64), (60, 64, 67)])
def test_large_planes_beside_a_small_box(ofm, ext):
    frags = [Fragment((2, 1, 3), ext, 2), Fragment((5, 9, 1), (9, 8, 7), 3)]
    wl = small_workload(tuple(e + 3 for e in ext), frags=frags, seed=6)
    H = O.hamiltonian(wl.grid, wl.V)
    ctx = ofm.Context()
    ctx.build_fragments(wl.grid, wl.V, frags, storage="fp32")
    eps, res, _ = ctx.fragment_eigs()
    assert res.max() <= 1e-5
    top = 12.0 / wl.grid.h ** 2 + np.abs(wl.V).max()
    for a, sl in ((0, slice(0, 2)), (1, slice(2, 5))):
        P = ctx.get_fragment_states(a)
        own = np.linalg.norm(O.fragment_hamiltonian(H, wl.grid, frags[a]) @ P - P * eps[sl], axis=0)
        assert np.all(np.abs(own - res[sl]) <= 0.02 * res[sl] + 6 * U32 * top)


@pytest.mark.parametrize("ext", [(2, 9, 10), (1, 12, 9), (9, 2, 10), (3, 8, 8), (10, 9, 1)])
def test_thin_boxes_along_their_longer_axes(ofm, ext):
    n = tuple(e + 3 for e in ext)
    _check(ofm, n, [Fragment((1, 2, 1), ext, 4), Fragment((0, 1, 2), ext, 2)], "fp32")

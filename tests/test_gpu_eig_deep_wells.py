"""FP32 fragment states where the potential has one deep narrow well: fragments
that do not hold it keep residuals at the level of their own Hamiltonian's
rounding, whatever its depth, and those that do converge too (the dense problem
of a block with one level tens of Ha below the rest).

Levels against the box's own Hamiltonian in FP64: within the residual's bound
1e-5 and a few FP32 roundings of |H| of that box."""
import numpy as np
import pytest

from ofm_inputs import Fragment, Grid, small_workload
from oracle import ofm_oracle as O

from gpu_util import U32, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


N = 26
FRAGS = [Fragment((0, 0, 0), (12, 12, 12), 8), Fragment((5, 2, 1), (11, 12, 10), 12),
         Fragment((13, 13, 13), (12, 11, 12), 8)]


@pytest.mark.parametrize("depth,at,holders", [(0.0, (6, 6, 6), ()), (20.0, (20, 19, 20), (2,)), (100.0, (20, 19, 20), (2,)),
                                              (20.0, (7, 6, 5), (0, 1)), (100.0, (7, 6, 5), (0, 1)),
                                              (1000.0, (25, 25, 25), ())])
def test_one_deep_narrow_well(ofm, depth, at, holders):
    wl = small_workload((N, N, N), frags=FRAGS, seed=4)
    V = wl.V.reshape(N, N, N).copy()   # [z][y][x]
    V[at[2], at[1], at[0]] -= depth
    H = O.hamiltonian(wl.grid, V.reshape(wl.V.shape))
    ctx = ofm.Context()
    ctx.build_fragments(wl.grid, V.reshape(wl.V.shape), FRAGS, storage="fp32")
    eps, res, _ = ctx.fragment_eigs()
    k = 0
    for a, f in enumerate(FRAGS):
        e, r = eps[k:k + f.n_states], res[k:k + f.n_states]
        k += f.n_states
        want = np.linalg.eigvalsh(O.fragment_hamiltonian(H, wl.grid, f).toarray())[:f.n_states]
        top = 12.0 / wl.grid.h ** 2 + np.abs(wl.V).max() + (depth if a in holders else 0.0)
        assert np.max(np.abs(e - want)) <= 1e-5 + 8 * U32 * top
        assert r.max() <= 1e-5

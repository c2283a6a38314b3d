"""FP32 fragment states of blocks with few wanted states: nothing among the
wanted levels bounds the filter's spread there, and a block whose guard vectors
are lost to the lowest state never settles.  Every start converges, in a few
passes' worth of launches, to the levels of the box's own Hamiltonian.

Tolerance: the residual's bound 1e-5 and a few FP32 roundings of |H|."""
import numpy as np
import pytest

from ofm_inputs import Fragment, small_workload
from oracle import ofm_oracle as O

from gpu_util import U32, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


@pytest.mark.parametrize("states", [1, 2, 3, 5])
def test_few_states_converge_from_every_start(ofm, states):
    frags = [Fragment((1, 1, 1), (11, 9, 8), states), Fragment((2, 3, 0), (8, 8, 6), max(1, states // 3))]
    wl = small_workload((15, 13, 12), frags=frags, seed=1)
    H = O.hamiltonian(wl.grid, wl.V)
    want = np.concatenate([np.linalg.eigvalsh(O.fragment_hamiltonian(H, wl.grid, f).toarray())[:f.n_states]
                           for f in frags])
    tol = 1e-5 + 8 * U32 * (12.0 / wl.grid.h ** 2 + np.abs(wl.V).max())
    ctx = ofm.Context()
    ctx.build_fragments(wl.grid, wl.V, frags, storage="fp32")
    for seed in range(24):
        eps, res, _ = ctx.fragment_eigs(seed=seed, max_iter=60)
        assert res.max() <= 1e-5
        assert np.max(np.abs(eps - want)) <= tol

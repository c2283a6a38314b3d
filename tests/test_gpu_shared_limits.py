"""Two contexts of one process whose plans need different amounts of shared
memory: a kernel's limit belongs to the kernel, so a smaller plan made in
between must not take it from the larger one's next call, which then gives
bitwise what it gave before."""
import numpy as np
import pytest

from ofm_inputs import Fragment, Grid, small_workload

from gpu_util import gpu_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


def _basis(ofm, n, ext, states, storage):
    frags = [Fragment((0, 0, 0), ext, states), Fragment((3, 2, 1), ext, states)]
    wl = small_workload(grid_n=(n, n, n), h=0.5, frags=frags, seed=7)
    ctx = ofm.Context()
    ctx.build_fragments(wl.grid, wl.V, wl.frags, storage=storage)
    return ctx


@pytest.mark.parametrize("storage,wide", [("fp32", 96), ("fp64", 60)])
def test_eigensolver_after_a_smaller_plan(ofm, storage, wide):
    big = _basis(ofm, 16, (12, 12, 12), wide, storage)
    first = big.fragment_eigs(max_iter=2, allow_not_converged=True)[0].copy()
    small = _basis(ofm, 10, (6, 5, 4), 3, storage)
    small.fragment_eigs(max_iter=2, allow_not_converged=True)
    assert np.array_equal(big.fragment_eigs(max_iter=2, allow_not_converged=True)[0], first)


def test_staged_stencil_after_a_smaller_plan(ofm, monkeypatch):
    monkeypatch.setenv("OFM_STENCIL", "staged")
    out = []
    ctxs = []
    for n, ext, states in ((16, (14, 12, 12), 96), (10, (6, 5, 4), 3)):
        ctx = _basis(ofm, n, ext, states, "fp32")
        rng = np.random.default_rng(states)
        for a in range(2):
            ctx.set_fragment_states(a, rng.standard_normal((int(np.prod(ext)), states)).astype(np.float32).astype(float))
        ctxs.append(ctx)
    for ctx in (ctxs[0], ctxs[1], ctxs[0]):
        ctx.assemble("fp32", schedule="pair", use_graph=False)
        out.append(ctx.get_blocks().copy())
    assert np.array_equal(out[0], out[2])

"""The CUDA-core contraction's register tiles at their edges: state counts
around one register tile, one 64-wide output tile and its multiples, uneven
between the two fragments, in FP64 and FP32, against the oracle; the Gram of
the FP64 eigensolver (upper half only) and the pencil product's row and
column tiles."""
import numpy as np
import pytest

from ofm_inputs import Fragment, random_states, small_workload
from oracle import ofm_oracle as O

from gpu_util import U32, U64, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


def _two(na, nb):
    frags = [Fragment((0, 0, 0), (11, 7, 6), na), Fragment((5, 3, 2), (9, 5, 7), nb)]
    return small_workload((20, 13, 12), frags=frags)


@pytest.mark.parametrize("na,nb", [(1, 1), (1, 64), (2, 3), (6, 6), (21, 21), (33, 31), (64, 1),
                                   (65, 32), (63, 66), (128, 130)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_pair_blocks_at_tile_edges(ofm, na, nb, prec):
    wl = _two(na, nb)
    H = O.hamiltonian(wl.grid, wl.V)
    Phis = [random_states(wl.grid, f, 7 + i).astype(np.float32).astype(np.float64)
            for i, f in enumerate(wl.frags)]
    ctx = ofm.Context()
    ctx.build_fragments(wl.grid, wl.V, wl.frags, storage=prec)
    for a, P in enumerate(Phis):
        ctx.set_fragment_states(a, P)
    ctx.assemble(prec, schedule="pair")
    u = U64 if prec == "fp64" else U32
    hn = 12.0 / wl.grid.h ** 2 + np.abs(wl.V).max()   # bound of |H phi| and of its terms
    for a, b in ((0, 0), (0, 1), (1, 1)):
        Hw, Sw = O.pair_block(H, wl.grid, wl.frags[a], Phis[a], wl.frags[b], Phis[b])
        if a == b:
            Hw, Sw = 0.5 * (Hw + Hw.T), 0.5 * (Sw + Sw.T)
        Hg, Sg = ctx.block(a, b)
        K = int(np.prod(wl.frags[b].ext)) * 2 + 32
        norm = np.linalg.norm(Phis[a], axis=0)[:, None] * np.linalg.norm(Phis[b], axis=0)[None]
        assert np.all(np.abs(Sg - Sw) <= K * u * norm)
        assert np.all(np.abs(Hg - Hw) <= K * u * hn * norm)


@pytest.mark.parametrize("n", [1, 5, 52, 60])
def test_fp64_eigenvalues_at_gram_tile_edges(ofm, n):
    # blocks of n + max(4, n / 4) vectors: 5, 9, 65 and 75
    wl = small_workload((18, 9, 9), frags=[Fragment((2, 1, 1), (12, 7, 7), n)])
    H = O.hamiltonian(wl.grid, wl.V)
    want = O.fragment_eigs(H, wl.grid, wl.frags[0])[0]
    ctx = ofm.Context()
    ctx.build_fragments(wl.grid, wl.V, wl.frags, storage="fp64")
    eps, res, _ = ctx.fragment_eigs()
    assert res.max() <= 1e-9
    assert np.max(np.abs(eps - want)) < 1e-9


@pytest.mark.parametrize("states", [1, 7, 16, 37, 70])
def test_pencil_tiles(ofm, states):
    import torch
    frags = [Fragment((4 * i, 0, 0), (8, 8, 8), states + i) for i in range(3)]
    wl = small_workload((24, 8, 8), frags=frags)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = ofm.Context(stream)
        ctx.build_fragments(wl.grid, wl.V, wl.frags, storage="fp64")
        for a, f in enumerate(wl.frags):
            ctx.set_fragment_states(a, random_states(wl.grid, f, 3 + a))
        ctx.assemble("fp64")
        Hd, Sd = ctx.dense_HS()
        n = Hd.shape[0]
        for k in (1, 2, 3, 15, 16, 17, 33):
            X = np.random.default_rng(k).standard_normal((k, n))
            Xd = torch.from_numpy(X).cuda()
            for which, M in (("H", Hd), ("S", Sd)):
                Y = ctx.pencil_apply(which, Xd)
                stream.synchronize()
                scale = (n + 8) * U64 * (np.abs(X) @ np.abs(M).T)
                assert np.all(np.abs(Y.cpu().numpy() - X @ M.T) <= scale), (k, which)

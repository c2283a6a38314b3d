"""The pair schedule's packed operands at their edges: box edges and overlaps
that start and end inside a group of eight points, overlaps of one point
column, boxes that wrap or span the cell, state counts around one and several
output tiles, in the three operand types, against the oracle; and a captured
assembly whose operand buffer is re-allocated by another schedule.

Bounds as in test_gpu_tensorcore.check_blocks (rounded inputs, FP32 sums), but
with the unit roundoff of BF16's eight significant bits, 2^-8: overlaps of a few
points reach what longer sums average out."""
import numpy as np
import pytest

from ofm_inputs import Fragment, Grid, small_workload
from oracle import ofm_oracle as O

from gpu_util import gpu_lib
import test_gpu_tensorcore
from test_gpu_tensorcore import check_blocks, fp32_states

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


@pytest.fixture(autouse=True)
def bf16_roundoff(monkeypatch):
    monkeypatch.setitem(test_gpu_tensorcore.U_IN, "bf16", 2.0 ** -8)


GEOMS = {
    # x offsets 1..7 within a group, an overlap of one column, n0 = 21
    "offsets": (Grid((21, 9, 8), 0.45), [Fragment((0, 0, 0), (9, 5, 5), 1), Fragment((7, 1, 2), (6, 7, 4), 15),
                                         Fragment((8, 4, 0), (11, 5, 8), 16), Fragment((3, 2, 3), (5, 4, 5), 17)]),
    # boxes over the cell's seam, one that spans it, one a point wide
    "seam": (Grid((19, 8, 9), 0.5), [Fragment((15, 0, 0), (9, 8, 5), 33), Fragment((0, 5, 4), (19, 6, 7), 31),
                                     Fragment((18, 7, 2), (1, 8, 9), 2), Fragment((12, 3, 8), (8, 1, 1), 5)]),
    # several output tiles, uneven
    "tiles": (Grid((40, 9, 9), 0.5), [Fragment((33, 1, 2), (20, 7, 6), 128), Fragment((3, 0, 0), (17, 9, 7), 64),
                                      Fragment((10, 2, 1), (13, 5, 7), 65), Fragment((20, 0, 3), (16, 9, 6), 127)]),
}


def _ctx(ofm, grid, V, frags, Phis):
    ctx = ofm.Context()
    ctx.build_fragments(grid, V, frags, storage="fp32")
    for a, P in enumerate(Phis):
        ctx.set_fragment_states(a, P)
    return ctx


@pytest.mark.parametrize("prec", ["tf32", "bf16", "bf16x3"])
@pytest.mark.parametrize("geom", sorted(GEOMS))
def test_pair_blocks_from_packed_operands(ofm, geom, prec):
    grid, frags = GEOMS[geom]
    wl = small_workload(grid_n=grid.n, h=grid.h, frags=frags, seed=11)
    Phis = fp32_states(grid, frags, 700)
    H = O.hamiltonian(grid, wl.V)
    ctx = _ctx(ofm, grid, wl.V, frags, Phis)
    ctx.assemble(prec, schedule="pair")
    check_blocks(ctx, wl, Phis, H, O.pair_list(grid, frags), prec)


def test_captured_pair_assembly_after_buffers_moved(ofm):
    grid, frags = GEOMS["tiles"]
    wl = small_workload(grid_n=grid.n, h=grid.h, frags=frags, seed=12)
    Phis = fp32_states(grid, frags, 710)
    ctx = _ctx(ofm, grid, wl.V, frags, Phis)
    H = O.hamiltonian(grid, wl.V)
    pairs = O.pair_list(grid, frags)
    # bf16 operands are the smallest: the later types and the other schedule make the buffers grow
    runs = [("bf16", "pair"), ("bf16x3", "region"), ("bf16", "pair"), ("tf32", "pair"), ("bf16x3", "region"),
            ("bf16", "pair")]
    first = {}
    for prec, sched in runs:
        ctx.assemble(prec, schedule=sched)
        got = [ctx.block(a, b) for a, b in pairs]
        check_blocks(ctx, wl, Phis, H, pairs, prec)
        for (g, w) in zip(got, first.setdefault((prec, sched), got)):
            assert np.array_equal(g[0], w[0]) and np.array_equal(g[1], w[1])

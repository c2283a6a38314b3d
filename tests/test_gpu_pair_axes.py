"""The pair schedule's operand units along each of the three axes: one set of
boxes, ragged against groups of eight points, over the cell's seam and spanning
it, laid out so that x, y and z in turn give the fewest units, in the three
operand types and in check mode, against the oracle; chains of overlapping boxes along
each axis; and BF16's half-size operands before and after the others'.

Bounds as in test_gpu_pair_planes (unit roundoff of BF16 2^-8)."""
import itertools

import numpy as np
import pytest

from ofm_inputs import Fragment, Grid, small_workload
from oracle import ofm_oracle as O

from gpu_util import gpu_lib
from test_gpu_pair_planes import _ctx, bf16_roundoff  # noqa: F401  (autouse fixture)
from test_gpu_tensorcore import check_blocks, fp32_states

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


def _turned(n, boxes, axes):
    turn = lambda v: tuple(v[a] for a in axes)
    return Grid(turn(n), 0.5), [Fragment(turn(o), turn(e), m) for o, e, m in boxes]


RAGGED = (21, 16, 19), [((3, 2, 15), (9, 6, 9), 17), ((7, 5, 0), (6, 7, 19), 9), ((18, 14, 18), (8, 8, 4), 33),
                        ((5, 9, 3), (11, 5, 8), 5)]
CHAIN = (28, 9, 8), [((7 * i + 1, 0, 0), (11, 9, 8), 6 + 9 * i) for i in range(4)]


@pytest.mark.parametrize("prec", ["tf32", "bf16", "bf16x3"])
@pytest.mark.parametrize("axes", list(itertools.permutations(range(3))))
@pytest.mark.parametrize("layout", ["ragged", "chain"])
def test_units_along_every_axis(ofm, layout, axes, prec):
    grid, frags = _turned(*(RAGGED if layout == "ragged" else CHAIN), axes)
    wl = small_workload(grid_n=grid.n, h=grid.h, frags=frags, seed=21)
    Phis = fp32_states(grid, frags, 810)
    ctx = _ctx(ofm, grid, wl.V, frags, Phis)
    ctx.set_checks(True)
    ctx.assemble(prec, schedule="pair")
    check_blocks(ctx, wl, Phis, O.hamiltonian(grid, wl.V), O.pair_list(grid, frags), prec)


def test_half_size_operands_between_others(ofm):
    grid, frags = _turned(*RAGGED, (2, 0, 1))
    wl = small_workload(grid_n=grid.n, h=grid.h, frags=frags, seed=22)
    ctx = _ctx(ofm, grid, wl.V, frags, fp32_states(grid, frags, 820))
    first = {}
    for prec in ("bf16", "bf16x3", "bf16", "tf32", "bf16", "bf16x3"):
        ctx.assemble(prec, schedule="pair")
        got = ctx.get_blocks()
        assert np.array_equal(got, first.setdefault(prec, got))

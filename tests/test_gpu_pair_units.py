"""The pair schedule's units in shared memory at the edges of their forms: state
counts whose stages hold three, four and more units of both fragments (a's units
whole or by parts), odd numbers of units with 8 to 256 MMA columns (the zero half
of the last K step), pairs of a fragment with itself, in the three operand types
and in check mode, against the oracle.

Bounds as in test_gpu_pair_planes."""
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


@pytest.mark.parametrize("prec", ["tf32", "bf16", "bf16x3"])
@pytest.mark.parametrize("states", [(8, 128), (96, 96), (96, 97), (104, 88), (128, 128), (121, 16), (1, 9)])
def test_units_whole_and_by_parts(ofm, states, prec):
    # boxes of 5 x 7 x 6 and 6 x 5 x 9 points: odd numbers of units along every axis
    grid = Grid((15, 11, 13), 0.5)
    frags = [Fragment((1, 2, 3), (5, 7, 6), states[0]), Fragment((4, 4, 1), (6, 5, 9), states[1]),
             Fragment((12, 8, 9), (9, 6, 7), 24)]
    wl = small_workload(grid_n=grid.n, h=grid.h, frags=frags, seed=31)
    Phis = fp32_states(grid, frags, 900)
    ctx = _ctx(ofm, grid, wl.V, frags, Phis)
    ctx.set_checks(True)
    ctx.assemble(prec, schedule="pair")
    check_blocks(ctx, wl, Phis, O.hamiltonian(grid, wl.V), O.pair_list(grid, frags), prec)

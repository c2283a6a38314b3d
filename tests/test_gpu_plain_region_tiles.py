"""The plain region contraction at the edges of its row blocks and column
quarters: stacked rows just below and above the counts where rows move from
spread to consecutive (32, 64, 96 and 128 rows), fragments that cross 16-row
blocks, and many fragments per region, whose pairs fill a triangle of the
stacked product.  Bounds as in test_gpu_plain_region."""
import numpy as np
import pytest

from ofm_inputs import Fragment, Grid, small_workload
from oracle import ofm_oracle as O

from gpu_util import gpu_lib
from test_gpu_plain_region import check, v32
from test_gpu_tensorcore import fp32_states

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


def _row(states):   # boxes along x, each overlapping its neighbours
    return Grid((8 * len(states), 7, 8), 0.5), [Fragment((8 * a, 0, 0), (16, 7, 8), n)
                                               for a, n in enumerate(states)]


def _cube(n):       # eight boxes that share a region, n stacked states each
    return Grid((20, 20, 20), 0.5), [Fragment((10 * i, 10 * j, 10 * k), (16, 15, 16), n + (i + j + k) % 2)
                                     for k in range(2) for j in range(2) for i in range(2)]


GEOMS = {"rows32": _row([8, 8, 16, 15]), "rows64": _row([33, 30, 34, 24]), "rows96": _row([49, 40, 41, 56]),
         "rows128": _row([63, 65, 64, 128]), "cube9": _cube(9), "cube45": _cube(45)}


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("geom", sorted(GEOMS))
def test_plain_region_blocks(ofm, geom, prec):
    grid, frags = GEOMS[geom]
    wl = small_workload(grid_n=grid.n, h=grid.h, frags=frags, seed=5)
    Phis = fp32_states(grid, frags, 640)
    H = O.hamiltonian(grid, v32(wl.V) if prec == "fp64" else wl.V)
    ctx = ofm.Context()
    ctx.build_fragments(grid, wl.V, frags, storage="fp32")
    for a, P in enumerate(Phis):
        ctx.set_fragment_states(a, P)
    ctx.assemble(prec, schedule="region")
    check(ctx, wl, Phis, H, O.pair_list(grid, frags), prec, "region")

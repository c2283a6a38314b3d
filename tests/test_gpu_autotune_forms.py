"""The autotuner of a tensor-core precision times one row of candidates: its pair
schedule runs no stencil kernel, so there is no form to choose, and the form that
an FP32 tuning chose stays the context's."""
import numpy as np
import pytest

from gpu_util import gpu_lib
from test_gpu_autotune import _check_bounds, _ctx, chain  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofm():
    return gpu_lib()


@pytest.mark.parametrize("prec", ["tf32", "bf16", "bf16x3"])
def test_one_form_for_the_tensor_cores(ofm, chain, prec):  # noqa: F811
    wl, Phis, H = chain
    ctx = _ctx(ofm, wl, Phis)
    _, form, ms, times = ctx.autotune_assembly(prec, chunks=[512, 1024], reps=2)
    assert form == 1 and np.all(times[0] > 0) and np.all(times[1] == -1.0)
    form32, times32 = ctx.autotune_assembly("fp32", chunks=[512], reps=2)[1::2]
    assert form32 in (1, 2) and times32[0, 0] > 0
    ctx.autotune_assembly(prec, chunks=[512], reps=1)
    ctx.assemble("fp32", schedule="pair")
    _check_bounds(ctx, wl, Phis, H, "fp32")

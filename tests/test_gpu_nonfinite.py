"""A NaN or +inf in a potential that a caller hands in is found, wherever it lies: at the edge of a window,
alone among pixels without mass, over a whole block, chunk or row."""
import numpy as np
import pytest

from paper_2512_19072_gb300 import inputs
from fot_testutil import f32, to_dev

pytestmark = pytest.mark.gpu


def _place(psi, where, val):
    psi = psi.copy()
    if where == "corner":
        psi[0, 0] = val
    elif where == "block":
        psi[37, 40:48] = val
    elif where == "chunk":
        psi[37, 32:64] = val
    elif where == "row":
        psi[37] = val
    elif where == "alone":
        psi[:] = -np.inf
        psi[10, 10], psi[37, 45] = 0.0, val
    return psi


# exact windows, 16- and 32-wide tiles; one kernel and two; aligned rows and not
@pytest.mark.parametrize("form", ["fp32", "mixed", "bf16"])
@pytest.mark.parametrize("shape,eps", [((64, 64), 1.0), ((64, 67), 16.0), ((700, 640), 3.0), ((600, 72), 200.0)])
@pytest.mark.parametrize("val", [np.nan, np.inf])
def test_nonfinite_potential_is_latched(fot_lib, form, shape, eps, val):
    B = fot_lib
    psi = inputs.random_potential(*shape, scale=0.02 * max(shape) ** 2 + 3 * eps, seed=8)
    ones = to_dev(np.ones(shape))
    for where in ("corner", "block", "chunk", "row", "alone"):
        ctx = B.fot_create(*shape, {"fp32": B.FOT_FP32, "mixed": B.FOT_MIXED, "bf16": B.FOT_BF16}[form])
        B.fot_set_problem(ctx, ones, ones)
        B.fot_u_update(ctx, to_dev(_place(psi, where, val)), eps)
        with pytest.raises(B.FotError) as err:
            B.fot_sync(ctx)
        assert B.STATUS[err.value.status] == "FOT_ENONFINITE", where
        ctx.close()


@pytest.mark.parametrize("eps", [1.0, 60.0])
def test_nonfinite_potential_shows_in_the_moments(fot_lib, eps):
    B = fot_lib
    psi = f32(inputs.random_potential(64, 64, scale=300.0, seed=9))
    ctx = B.fot_create(64, 64)
    for where in ("corner", "row", "alone"):
        _, Dx, Dy = B.fot_moments(ctx, to_dev(_place(psi, where, np.nan)), to_dev(np.zeros((64, 64))), eps, 0.4)
        assert not Dx.isfinite().all() and not Dy.isfinite().all(), where
    ctx.close()

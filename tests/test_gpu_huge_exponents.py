"""Potentials so large against eps that the rounding of an exponent (2^-24 of it) leaves the range of FP32
exponentials: updates stay finite and right to FP32 rounding of the potentials."""
import numpy as np
import pytest

from oracle import fot
from paper_2512_19072_gb300 import inputs
from fot_testutil import POT_RTOL, assert_pot_close, f32, to_dev, to_np

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:invalid value encountered")]


# exact windows, 16- and 32-wide products; one kernel and two (516); the last: beyond the plan's sentinel
@pytest.mark.parametrize("form", ["fp32", "mixed", "dense"])
@pytest.mark.parametrize("shape,eps,scale", [((40, 36), 1e-3, 1e7), ((40, 36), 16.0, 1e11), ((40, 36), 200.0, 1e13),
                                             ((9, 516), 1e-3, 1e8), ((9, 516), 60.0, 1e13), ((40, 36), 1.0, 2.5e38)])
def test_updates_at_huge_exponents(fot_lib, form, shape, eps, scale):
    B = fot_lib
    rng = np.random.default_rng(31)
    g, G = (f32(rng.uniform(0.05, 1.0, size=shape)) for _ in range(2))
    psi = f32(inputs.random_potential(*shape, scale=scale, seed=32, zero_frac=0.1))
    ctx = B.fot_create(*shape, {"fp32": B.FOT_FP32, "mixed": B.FOT_MIXED, "dense": B.FOT_FP32_DENSE}[form])
    B.fot_set_problem(ctx, to_dev(g), to_dev(G))
    f = to_np(B.fot_u_update(ctx, to_dev(psi), eps))
    B.fot_sync(ctx)
    ctx.close()
    assert_pot_close(f, fot.u_update(psi, fot.log0(fot.marginal(g)), eps)[0], rtol=POT_RTOL)

"""Errors of the kernel sums that FP32 rounding of the potentials hides: log-sums of potentials for
which the constants of a pass (log2(e) / eps and half of it) are exact in FP32 and the log-sums lie
near zero, so that what is left is the error of the sums themselves."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

LOG2E = 1.4426950408889634


def _level_potential(shape, eps, seed):
    """Noise about the level whose log-sum is zero."""
    gen = torch.Generator().manual_seed(seed)
    noise = 0.3 * eps * (torch.rand(shape, generator=gen) - 0.5)
    return (noise - eps * math.log(2 * math.pi * eps)).cuda()


def _logsum(B, precision, psi, eps):
    ctx = B.fot_create(*psi.shape, precision)
    B.fot_set_problem(ctx, torch.ones_like(psi), torch.ones_like(psi))
    _, S = B.fot_u_update(ctx, psi, eps, with_logsum=True)
    B.fot_sync(ctx)
    terms = B.fot_work_split(ctx)
    ctx.close()
    return S.double(), terms


@pytest.mark.parametrize("shape", [(256, 256), (600, 131)])
@pytest.mark.parametrize("power", [2.5, 4.0, 6.0])
def test_products_of_fp32_operands_are_not_biased(fot_lib, shape, power):
    """8-, 16- and 32-wide tiles, one-kernel and two-kernel passes, against the dense form, which has
    the same exponentials and no products.  Bound: the tensor core cuts a step's sum at 24 bits when
    it adds the last two products, 2^-24 on average each, so 2^-23 per pass and 2^-22 in two; the
    operands' parts are rounded and add nothing on average."""
    B = fot_lib
    eps = LOG2E * 2.0 ** power
    psi = _level_potential(shape, eps, 3)
    banded, terms = _logsum(B, B.FOT_FP32, psi, eps)
    dense, _ = _logsum(B, B.FOT_FP32_DENSE, psi, eps)
    assert terms[0] > 0 and terms[1] == 0                   # products alone
    assert abs((banded - dense).mean().item()) <= 2.0 ** -22

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
@pytest.mark.parametrize("power", [3.5, 5.0, 6.0, 7.0])
def test_products_of_fp32_operands_are_not_biased(fot_lib, shape, power):
    """16- and 32-wide tiles, one-kernel and two-kernel passes, against the dense form, which has
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


def _exact_logsum(psi, eps):
    """The same in 64 bits, in the units the kernels write (log2 times ln 2 as FP32 has it)."""
    def axis(x):
        i = torch.arange(x.shape[1], dtype=torch.float64, device=x.device)
        top = x.max(dim=1, keepdim=True).values
        return (torch.log(torch.exp(x - top) @ torch.exp(-(i[:, None] - i) ** 2 / (2 * eps))) + top).T
    ln2 = math.log(2)
    return axis(axis(psi.double() / eps)) * (torch.tensor(ln2, dtype=torch.float32).item() / ln2)


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("shape", [(1200, 900), (512, 508)])
def test_long_windows_keep_their_precision(fot_lib, shape, precision):
    """Windows of 70 steps (eps 5909; across the whole row at 512): the step scale's rounding, 2^-25, must
    not be carried through the walk (35 steps to the largest term: 1e-6).  Bound on the mean square where
    the log-sum is small, natural logarithm: per pass an operand's rounding (FP32: ex2 and the
    exponent, 2^-22; BF16 pairs: 2^-17 averaged over a step's 16 positions, 2^-19 at worst) and a rounding of
    the log-sum between the passes (its size is log(2 pi eps) / 2 = 5: 2^-22); twice that for both passes."""
    B = fot_lib
    eps = LOG2E * 2.0 ** 12
    psi = _level_potential(shape, eps, 4)
    got, _ = _logsum(B, {"fp32": B.FOT_FP32, "mixed": B.FOT_MIXED}[precision], psi, eps)
    ref = _exact_logsum(psi, eps)
    near = ref.abs() < 0.3
    rms = (got - ref)[near].pow(2).mean().sqrt().item()
    assert near.sum() > 1000
    assert rms <= (2 * 2.0 ** -22 + 2 * 2.0 ** -22 if precision == "fp32" else 2 * (2.0 ** -19 + 2.0 ** -22)), rms


@pytest.mark.parametrize("form", ["fp32", "mixed"])
def test_small_eps_sums_are_exact(fot_lib, form):
    """eps 8: one exponential per term and output, whatever the form.  Bound on the mean square, natural
    logarithm: per pass ex2's 2^-22, uniform, over sqrt(4 pi eps) = 10 terms that matter, and the rounding of a
    log-sum below 4 (2^-23, uniform); both passes, and half as much again for what is not random."""
    B = fot_lib
    eps = LOG2E * 2.0 ** 2.5
    psi = _level_potential((300, 256), eps, 5)
    got, terms = _logsum(B, {"fp32": B.FOT_FP32, "mixed": B.FOT_MIXED}[form], psi, eps)
    ref = _exact_logsum(psi, eps)
    near = ref.abs() < 0.3
    rms = (got - ref)[near].pow(2).mean().sqrt().item()
    assert near.sum() > 1000 and terms[0] == 0 and terms[2] == 0
    assert rms <= 1.5 * math.sqrt(2) * (2.0 ** -22 / math.sqrt(30) + 2.0 ** -23 * math.log(2) / math.sqrt(3)), rms

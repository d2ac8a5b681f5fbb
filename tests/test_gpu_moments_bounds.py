"""The moment passes (Eqs. 9-10) against the oracle within bounds of each axis's own pixel pitch, at the
edges of the kernels' units and at pitches of metres, where coordinates reach 10^5."""
import numpy as np
import pytest

from oracle import fot
from paper_2512_19072_gb300 import inputs
from fot_testutil import f32, to_dev, to_np

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:invalid value encountered")]


def _check(B, psi, S, eps, dx):
    """Each weight is the exponential of logarithms of size <= lmax, eight of whose FP32 roundings change it
    by d <= 8 2^-24 lmax, and passes through two products of 2^-21.  A sum over a window of positions
    p >= 0, of coordinates up to twice the largest apart, and its divisor both move by that."""
    rows, cols = psi.shape
    ctx = B.fot_create(rows, cols)
    _, Dx, Dy = (to_np(t) for t in B.fot_moments(ctx, to_dev(psi), to_dev(S), eps, dx))
    ctx.close()
    with np.errstate(over="ignore"):
        Dx_r, Dy_r = fot.moments(psi, S, eps, dx)
    S_psi = fot.log_kernel_apply(psi, eps)
    lmax = np.abs(S).max() + np.abs(psi[np.isfinite(psi)]).max() / eps
    bound = 2 * (np.expm1(2 * 8 * 2.0 ** -24 * lmax) + 4 * 2.0 ** -21) * np.exp(S_psi - S)
    for got, ref, n in ((Dx, Dx_r, rows), (Dy, Dy_r, cols)):
        coord = max(n // 2, 1) / (n * dx)
        assert (np.abs(got - ref) <= bound * coord).all(), ((np.abs(got - ref) / (bound * coord)).max(), n)


# exact windows, 16-wide products, rows longer than the staging buffer
@pytest.mark.parametrize("shape,eps", [((7, 129), 1.5), ((33, 66), 20.0), ((65, 40), 300.0), ((10, 1499), 1e5),
                                       ((1499, 10), 1e5), ((40, 700), 500.0)])
def test_moments_within_each_axis_bound(fot_lib, shape, eps):
    psi = f32(inputs.random_potential(*shape, scale=0.02 * max(shape) ** 2 + 3 * eps, seed=8, zero_frac=0.15))
    S = f32(fot.log_kernel_apply(psi, eps) + np.random.default_rng(9).normal(0, 0.2, size=shape))
    _check(fot_lib, psi, S, eps, 0.41)


# steep potentials: the offset lies up to 2^100 below the sums that the coordinates multiply
@pytest.mark.parametrize("n,eps,dx", [(64, 1.0, 8e-6), (61, 1.0, 8e-6), (96, 2.0, 1e-9), (96, 40.0, 8e-6)])
def test_moments_at_a_small_pitch(fot_lib, n, eps, dx):
    psi = f32(np.random.default_rng(4).random((n, n)) * 100 * eps)
    S = f32(fot.log_kernel_apply(psi, eps))
    _check(fot_lib, psi, S, eps, dx)

"""Paths that ordinary sizes do not take: two problems per launch with plan and sums apart, transforms of the
longest lines, units summed in segments or exactly because their windows span a gap."""
import numpy as np
import pytest

from oracle import fot
from paper_2512_19072_gb300 import inputs
from fot_testutil import POT_RTOL, assert_pot_close, f32, to_dev, to_np
from test_gpu_cfot import _beam, _conv_rel_error
from test_gpu_intensity import _bound

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:invalid value encountered",
                                                          "ignore:divide by zero")]


@pytest.mark.parametrize("form", ["fp32", "mixed"])
@pytest.mark.parametrize("shape,eps", [((24, 532), 600.0), ((530, 21), 600.0), ((20, 600), 40.0), ((516, 516), 900.0)])
def test_backward_with_a_side_above_512(fot_lib, form, shape, eps):
    """The adjoint's pair passes with plan and sums apart, against the dense form.  Bound: exponents reach
    C / eps, so one FP32 rounding of an exponent is C / eps 2^-24 relative, in each of ten half-steps and of
    their transposes, on both sides; mixed products add 2^-15 to each."""
    B = fot_lib
    rng = np.random.default_rng(51)
    g, G = (to_dev(f32(rng.uniform(0.3, 1.0, size=shape))) for _ in range(2))
    seeds = [to_dev(f32(rng.normal(size=shape))) for _ in range(3)]
    grads = {}
    for name, P in (("dense", B.FOT_FP32_DENSE), (form, {"fp32": B.FOT_FP32, "mixed": B.FOT_MIXED}[form])):
        ctx = B.fot_create(*shape, P)
        B.fot_solve(ctx, g, G, [eps], 5, dx=0.1)
        grads[name] = [to_np(t) for t in B.fot_backward(ctx, g, G, *seeds, checkpoint_every=2)]
        ctx.close()
    tol = 2 * 20 * (max(shape) ** 2 / (2 * eps) * 2.0 ** -24) + (20 * 2.0 ** -15 if form == "mixed" else 0.0)
    assert tol < 2e-2
    for got, ref in zip(grads[form], grads["dense"]):
        assert np.abs(got - ref).max() <= tol * np.abs(ref).max(), np.abs(got - ref).max() / np.abs(ref).max()


@pytest.mark.parametrize("shape", [(2048, 4), (4, 2048), (8, 4096), (4096, 16), (2048, 256)])
def test_far_field_of_the_longest_lines(fot_lib, shape):
    B = fot_lib
    rng = np.random.default_rng(52)
    g, G = (f32(rng.uniform(0.1, 1.0, shape)) for _ in range(2))
    phi = f32(rng.normal(0.0, 3.0, shape))
    ctx = B.fot_create(*shape)
    B.fot_set_problem(ctx, to_dev(g), to_dev(G))
    loss, inten = B.fot_intensity_loss(ctx, to_dev(phi), with_intensity=True)
    ctx.close()
    ref, iref = fot.intensity_loss(g, phi, G)
    tol = _bound(shape, g)
    assert abs(loss - ref) <= tol and np.abs(to_np(inten) - iref).max() <= tol
    assert np.abs(to_np(inten) - iref).max() <= 2e-4 * iref.max()   # (every pixel, not the sum's share of one)


@pytest.mark.parametrize("shape,eps", [((1100, 6), 1.2e5), ((5, 2048), 4e5), ((600, 9), 4e4)])
def test_convolutions_of_the_longest_lines(fot_lib, shape, eps):
    """As test_cfot_matches_oracle, padded to 2048 and 4096."""
    B = fot_lib
    iters = 3
    g = _beam(*shape, 0.45 * shape[0], 0.55 * shape[1], max(shape) / 5, 1.0)
    G = _beam(*shape, 0.55 * shape[0], 0.40 * shape[1], max(shape) / 4, 1.0)
    d = _conv_rel_error(np.full(shape, 1.0 / (shape[0] * shape[1])), eps)
    for t in range(1, iters + 1):
        u, V, _ = fot.cfot_iterate(g, G, eps, t)
        d = max(d, _conv_rel_error(u, eps), _conv_rel_error(V, eps))
    lm = max(np.abs(np.log(fot.marginal(x))).max() for x in (g, G))
    lu = max(np.abs(np.log(u)).max(), np.abs(np.log(V)).max())
    bound = 2 * iters * (d + 2.0 ** -24 * (lm + 4)) + 2.0 ** -24 * (lu + 1)
    assert bound < 1e-2
    ctx = B.fot_create(*shape)
    B.fot_cfot_solve(ctx, to_dev(g), to_dev(G), eps, iters)
    f, psi = B.fot_potentials(ctx)
    ctx.close()
    assert np.abs(to_np(f) - eps * np.log(u)).max() <= eps * bound
    assert np.abs(to_np(psi) - eps * np.log(V)).max() <= eps * bound


# two far-apart plateaus of equal height at the ends of each row: windows span the gap (as
# test_windows_across_a_gap), in one kernel (500) and in two; FP32 products in BF16 contexts whose rows are
# aligned are the segments
@pytest.mark.parametrize("form", ["fp32", "mixed", "bf16"])
@pytest.mark.parametrize("n,eps", [(500, 100.0), (640, 100.0), (500, 60.0)])
def test_units_across_a_gap_are_cut(fot_lib, form, n, eps):
    B = fot_lib
    k = np.arange(n, dtype=np.float64)
    row = np.full(n, -np.inf)
    row[:24] = 0.5 * (n / 2 - k[:24]) ** 2
    row[-24:] = 0.5 * (n / 2 - k[-24:]) ** 2
    psi = f32(np.stack([row + 0.3 * eps * i for i in range(12)]))
    g = f32(np.random.default_rng(53).uniform(0.05, 1.0, size=psi.shape))
    ctx = B.fot_create(*psi.shape, {"fp32": B.FOT_FP32, "mixed": B.FOT_MIXED, "bf16": B.FOT_BF16}[form])
    B.fot_set_problem(ctx, to_dev(g), to_dev(g))
    f = to_np(B.fot_u_update(ctx, to_dev(psi), eps))
    B.fot_sync(ctx)
    gemm, exact, tensor, _ = B.fot_work_split(ctx)
    ctx.close()
    assert gemm > 0 and exact == 0 and (tensor > 0) == (form != "fp32")
    ref, _ = fot.u_update(psi, fot.log0(fot.marginal(g)), eps)
    fin = np.isfinite(ref)
    assert np.array_equal(np.isneginf(f), np.isneginf(ref))
    # (form bounds per half-step: fot.h)
    tol = POT_RTOL * np.abs(ref[fin]).max() + {"fp32": 0.0, "mixed": 2.0 ** -15, "bf16": 2.0 ** -6}[form] * eps
    assert np.abs(f[fin] - ref[fin]).max() <= tol


# exponents whose rounding alone leaves the range of FP32 send a unit of products to exact sums
@pytest.mark.parametrize("cols", [36, 516])
def test_units_of_products_summed_exactly(fot_lib, cols):
    B = fot_lib
    psi = f32(inputs.random_potential(12, cols, scale=2.5e38, seed=54))
    g = f32(np.random.default_rng(55).uniform(0.05, 1.0, size=psi.shape))
    eps = 16.0
    psi = f32(np.clip(psi * 8.0, -3e38, 3e38))
    ctx = B.fot_create(*psi.shape)
    B.fot_set_problem(ctx, to_dev(g), to_dev(g))
    f = to_np(B.fot_u_update(ctx, to_dev(psi), eps))
    B.fot_sync(ctx)
    _, exact, _, _ = B.fot_work_split(ctx)
    ctx.close()
    assert exact > 0
    assert_pot_close(f, fot.u_update(psi, fot.log0(fot.marginal(g)), eps)[0], rtol=POT_RTOL)

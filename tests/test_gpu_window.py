"""The window sums of the banded passes at the edges of their units: half-steps against the FP64
oracle where tiles, row groups and windows end raggedly, where an item's rows do not fit its
staging buffer, where 32-wide units have to be cut or summed exactly, and where a potential's
steps put the plan's offsets far below the exact maxima.

Tolerances as in test_gpu_parity: FP32 rounding of the potentials (POT_RTOL), plus 2^-15 eps for
the split-BF16 form (two passes, each product within 2^-16)."""
import numpy as np
import pytest

from oracle import fot
from paper_2512_19072_gb300 import inputs
from fot_testutil import POT_RTOL, f32, to_dev, to_np

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:invalid value encountered")]


def _check(B, prec, psi, eps, seed):
    shape = psi.shape
    rng = np.random.default_rng(seed)
    g = f32(rng.uniform(0.05, 1.0, size=shape))
    G = f32(rng.uniform(0.05, 1.0, size=shape))
    g[rng.uniform(size=shape) < 0.1] = 0.0
    g[-1, -1] = 0.5
    ctx = B.fot_create(*shape, {"fp32": B.FOT_FP32, "mixed": B.FOT_MIXED}[prec])
    B.fot_set_problem(ctx, to_dev(g), to_dev(G))
    f = to_np(B.fot_u_update(ctx, to_dev(psi), eps))
    B.fot_sync(ctx)
    ctx.close()
    ref, _ = fot.u_update(psi, fot.log0(fot.marginal(g)), eps)
    fin = np.isfinite(ref)
    assert np.array_equal(np.isneginf(f), np.isneginf(ref))
    tol = POT_RTOL * np.abs(ref[fin]).max() + (2.0 ** -15 * eps if prec == "mixed" else 0.0)
    err = np.abs(f[fin] - ref[fin]).max()
    assert err <= tol, (err, tol)


# rows and columns around multiples of the row group (8), the tiles (16, 32) and the four tiles of
# an item, aligned and unaligned; eps for exact windows, 16-wide and 32-wide units
@pytest.mark.parametrize("prec", ["fp32", "mixed"])
@pytest.mark.parametrize("shape", [(7, 129), (9, 127), (33, 64), (65, 66), (24, 1)])
@pytest.mark.parametrize("eps", [1.5, 20.0, 400.0])
def test_ragged_units(fot_lib, prec, shape, eps):
    psi = f32(inputs.random_potential(*shape, scale=0.3 * max(shape) ** 2 + 3 * eps, seed=5, zero_frac=0.15))
    _check(fot_lib, prec, psi, eps, 1)


# passes of one kernel and of two: both sides of the longest row of a one-kernel product (512), row
# groups whose tiles divide unevenly among CTAs, exact rows with more tiles than warps (16), and
# two-kernel passes with ragged units
@pytest.mark.parametrize("prec", ["fp32", "mixed"])
@pytest.mark.parametrize("shape,eps", [((9, 512), 30.0), ((512, 9), 9.0), ((17, 511), 100.0), ((513, 12), 30.0),
                                       ((7, 545), 400.0), ((530, 3), 9.0), ((3, 1025), 1.5), ((1, 260), 0.7),
                                       ((2, 2050), 3.0)])
def test_one_and_two_kernel_passes(fot_lib, prec, shape, eps):
    psi = f32(inputs.random_potential(*shape, scale=0.1 * max(shape) ** 2 + 3 * eps, seed=12, zero_frac=0.15))
    _check(fot_lib, prec, psi, eps, 4)


# a batch whose passes are all exact, all products, or of both kinds gives what single solves give
@pytest.mark.parametrize("prec", ["fp32", "mixed"])
@pytest.mark.parametrize("shapes,eps", [([(40, 33)], [1.0]), ([(40, 33), (64, 64), (9, 130)], [1.0, 2.0, 1.5]),
                                        ([(40, 33), (600, 30)], [40.0, 60.0]),
                                        ([(40, 33), (64, 64), (600, 30)], [1.0, 40.0, 2.0])])
def test_batches_of_exact_and_product_problems(fot_lib, prec, shapes, eps):
    B = fot_lib
    P = {"fp32": B.FOT_FP32, "mixed": B.FOT_MIXED}[prec]
    rng = np.random.default_rng(13)
    gs = [to_dev(f32(rng.uniform(0.05, 1.0, size=s))) for s in shapes]
    Gs = [to_dev(f32(rng.uniform(0.05, 1.0, size=s))) for s in shapes]
    batch = B.fot_batch_create(shapes, P)
    B.fot_batch_solve(batch, gs, Gs, np.repeat(np.asarray(eps)[:, None], 4, axis=1), 4)
    for q, s in enumerate(shapes):
        ctx = B.fot_create(*s, P)
        B.fot_solve(ctx, gs[q], Gs[q], [eps[q]], 4)
        for a, b in zip(B.fot_potentials(B.fot_batch_context(batch, q)), B.fot_potentials(ctx)):
            assert np.array_equal(to_np(a), to_np(b)), q       # the same arithmetic
        ctx.close()
    batch.close()


# windows over whole rows of 1500 and 1499: more than an item's staging buffer holds
@pytest.mark.parametrize("prec", ["fp32", "mixed"])
@pytest.mark.parametrize("shape", [(10, 1500), (10, 1499)])
def test_rows_beyond_the_staging_buffer(fot_lib, prec, shape):
    psi = f32(inputs.random_potential(*shape, scale=2e4, seed=6))
    _check(fot_lib, prec, psi, 1e5, 2)


# two far-apart plateaus of equal height: the maximum jumps across the row within a tile, so the
# window spans the gap and the operands leave the tilted product's range
@pytest.mark.parametrize("prec", ["fp32", "mixed"])
@pytest.mark.parametrize("n,eps", [(640, 100.0), (641, 60.0), (640, 8.0)])
def test_windows_across_a_gap(fot_lib, prec, n, eps):
    k = np.arange(n, dtype=np.float64)
    row = np.full(n, -np.inf)
    row[:24] = 0.5 * (n / 2 - k[:24]) ** 2                 # the two ends tie at the centre
    row[-24:] = 0.5 * (n / 2 - k[-24:]) ** 2
    psi = np.stack([row + 0.3 * eps * i for i in range(12)])
    _check(fot_lib, prec, f32(psi), eps, 3)


# the moment passes at the same edges, against the oracle's moments; tolerance as in
# test_moments_kernel_matches_oracle (FP32 rounding of the logarithms, times the largest coordinate)
@pytest.mark.parametrize("shape,eps", [((7, 129), 1.5), ((33, 66), 20.0), ((65, 40), 300.0), ((10, 1499), 1e5)])
def test_moments_at_unit_edges(fot_lib, shape, eps):
    B = fot_lib
    psi = f32(inputs.random_potential(*shape, scale=0.02 * max(shape) ** 2 + 3 * eps, seed=8, zero_frac=0.15))
    S = f32(fot.log_kernel_apply(psi, eps) + np.random.default_rng(9).normal(0, 0.2, size=shape))
    dx = 0.41
    ctx = B.fot_create(*shape)
    _, Dx, Dy = (to_np(t) for t in B.fot_moments(ctx, to_dev(psi), to_dev(S), eps, dx))
    ctx.close()
    Dx_r, Dy_r = fot.moments(psi, S, eps, dx)
    lmax = (np.abs(S).max() + np.abs(psi[np.isfinite(psi)]).max() / eps) / np.log(2)
    cmax = max(shape) / 2 / (min(shape) * dx)
    tol = 4 * 2.0 ** -24 * lmax * cmax + 1e-6 * max(np.abs(Dx_r).max(), np.abs(Dy_r).max())
    assert np.abs(Dx - Dx_r).max() <= tol and np.abs(Dy - Dy_r).max() <= tol


# unequal grids: half-integer shifts, an output axis longer or shorter than the input axis, exact
# windows and 16- and 32-wide units; FP32 rounding of the potentials over the iterations
@pytest.mark.parametrize("shape_in,shape_out,eps", [((40, 51), (57, 36), 2.0), ((33, 130), (96, 23), 25.0),
                                                    ((70, 64), (64, 203), 500.0)])
def test_unequal_grids_at_unit_edges(fot_lib, shape_in, shape_out, eps):
    from oracle import rect
    from fot_testutil import solve_rtol
    rng = np.random.default_rng(12)
    g = f32(rng.uniform(0.05, 1.0, size=shape_in))
    G = f32(rng.uniform(0.05, 1.0, size=shape_out))
    G[rng.uniform(size=shape_out) < 0.2] = 0.0
    iters = 6
    f, psi = (to_np(t) for t in fot_lib.fot_solve_rect(to_dev(g), to_dev(G), [eps], iters))
    r = rect.fot_iterate_rect(g, G, eps, iters)
    for got, ref in ((f, r["f"]), (psi, r["psi"])):
        fin = np.isfinite(ref)
        assert np.array_equal(np.isneginf(got), np.isneginf(ref))
        assert np.abs(got[fin] - ref[fin]).max() <= solve_rtol(iters) * np.abs(ref[fin]).max()

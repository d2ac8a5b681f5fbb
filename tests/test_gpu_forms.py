"""Which passes of FOT_MIXED and FOT_BF16 contexts take BF16 operands: rows that are 16-byte aligned do,
the others keep FP32 operands and FP32 errors."""
import numpy as np
import pytest

from oracle import fot
from paper_2512_19072_gb300 import inputs
from fot_testutil import POT_RTOL, assert_pot_close, f32, to_dev, to_np

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:invalid value encountered")]


# neither side a multiple of 4: every pass in FP32, in one kernel and in two
@pytest.mark.parametrize("form", ["mixed", "bf16"])
@pytest.mark.parametrize("shape,eps", [((91, 66), 35.0), ((30, 531), 200.0)])
def test_unaligned_rows_keep_fp32_operands(fot_lib, form, shape, eps):
    B = fot_lib
    rng = np.random.default_rng(21)
    g, G = (f32(rng.uniform(0.05, 1.0, size=shape)) for _ in range(2))
    psi = f32(inputs.random_potential(*shape, scale=0.05 * max(shape) ** 2, seed=22, zero_frac=0.1))
    ctx = B.fot_create(*shape, {"mixed": B.FOT_MIXED, "bf16": B.FOT_BF16}[form])
    B.fot_set_problem(ctx, to_dev(g), to_dev(G))
    f = to_np(B.fot_u_update(ctx, to_dev(psi), eps))
    B.fot_sync(ctx)
    gemm, _, tensor, _ = B.fot_work_split(ctx)
    ctx.close()
    assert gemm > 0 and tensor == 0
    assert_pot_close(f, fot.u_update(psi, fot.log0(fot.marginal(g)), eps)[0], rtol=POT_RTOL)


# a batch of aligned and unaligned problems, and of both kinds of pass in one problem, gives what
# single solves give
def test_batch_of_aligned_and_unaligned_rows(fot_lib):
    B = fot_lib
    rng = np.random.default_rng(23)
    shapes, eps = [(64, 64), (63, 65), (64, 66), (90, 520), (31, 40)], [60.0, 40.0, 50.0, 200.0, 1.5]
    gs, Gs = ([to_dev(f32(rng.uniform(0.05, 1.0, size=s))) for s in shapes] for _ in range(2))
    batch = B.fot_batch_create(shapes, B.FOT_MIXED)
    B.fot_batch_solve(batch, gs, Gs, np.repeat(np.asarray(eps)[:, None], 3, axis=1), 3)
    for q, s in enumerate(shapes):
        ctx = B.fot_create(*s, B.FOT_MIXED)
        B.fot_solve(ctx, gs[q], Gs[q], [eps[q]], 3)
        for a, b in zip(B.fot_potentials(B.fot_batch_context(batch, q)), B.fot_potentials(ctx)):
            assert np.array_equal(to_np(a), to_np(b)), q
        assert (B.fot_work_split(ctx)[2] > 0) == (q in (0, 2, 3))   # some pass along a multiple of 4, eps large enough
        ctx.close()
    batch.close()

"""The sums of the intensity loss by themselves: a plane wave's far field is one pixel exactly, and a target of
N equal pixels elsewhere has b = exp(log b) with log b the FP32 logarithm of 1/N, so that the loss is known
to the last bit but for the arithmetic of the sum."""
import math

import numpy as np
import pytest

from fot_testutil import to_dev

pytestmark = pytest.mark.gpu

N = 64


def test_loss_of_equal_pixels(fot_lib):
    """Bound: exponentials of 2^-37 and pairs of FP32 numbers (2^-47) in every pixel, all the same way: 2^-36
    of the sum."""
    B = fot_lib
    ctx = B.fot_create(N, N)
    order = np.random.default_rng(41).permutation(N * N)
    order = order[order != N // 2 * N + N // 2]             # (the far field's pixel stays dark)
    phi, g = to_dev(np.zeros((N, N))), to_dev(np.ones((N, N)))
    for count in sorted({int(round(1.3 ** k)) for k in range(1, 32)} | {4095}):
        G = np.zeros(N * N)
        G[order[:count]] = 1.0
        B.fot_set_problem(ctx, g, to_dev(G.reshape(N, N)))
        loss = B.fot_intensity_loss(ctx, phi)
        want = 1.0 + count * math.exp(-float(np.float32(math.log(count))))
        assert abs(loss - want) <= 2.0 ** -36 * want, (count, loss / want - 1.0)
    ctx.close()

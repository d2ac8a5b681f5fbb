"""fot_cfot_solve returns before the work that its stream still has in front of it is done."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_first_cfot_solve_does_not_wait_for_its_stream(fot_lib):
    B = fot_lib
    g = torch.rand(96, 80, device="cuda", generator=torch.Generator("cuda").manual_seed(2)) + 0.5
    ref = B.fot_create(96, 80)
    B.fot_cfot_solve(ref, g, g, [900.0], 5)
    want = B.fot_potentials(ref)
    B.fot_sync(ref)
    ctx = B.fot_create(96, 80)
    torch.cuda.synchronize()
    before = torch.cuda.Event()
    torch.cuda._sleep(1_000_000_000)                        # about half a second
    before.record()
    B.fot_cfot_solve(ctx, g, g, [900.0], 5)
    assert not before.query()
    for a, b in zip(B.fot_potentials(ctx), want):
        assert torch.equal(a, b)
    ref.close()
    ctx.close()

"""Half-steps captured into a caller's CUDA graph: what they leave in the context (the BF16 forms' operand
tables) must not be taken for written before a replay, nor for unchanged after one."""
import pytest
import torch

pytestmark = pytest.mark.gpu

N = 64


@pytest.mark.parametrize("form", ["mixed", "bf16", "fp32"])
def test_captured_and_direct_updates_in_any_order(fot_lib, form):
    B = fot_lib
    P = {"mixed": B.FOT_MIXED, "bf16": B.FOT_BF16, "fp32": B.FOT_FP32}[form]
    ones = torch.ones(N, N, device="cuda")
    psi = 100.0 * torch.rand(N, N, device="cuda", generator=torch.Generator("cuda").manual_seed(1))

    def context():
        c = B.fot_create(N, N, P)
        B.fot_set_problem(c, ones, ones)
        B.fot_sync(c)
        return c

    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        want = {}
        for eps in (60.0, 100.0, 250.0):
            c = context()
            want[eps] = B.fot_u_update(c, psi, eps)
            B.fot_sync(c)
            c.close()

        def direct(c, eps):
            f = B.fot_u_update(c, psi, eps)
            B.fot_sync(c)
            assert torch.equal(f, want[eps]), eps

        c = context()
        direct(c, 100.0)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            f = B.fot_u_update(c, psi, 60.0)

        def replay():
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(f, want[60.0])

        direct(c, 60.0)                                     # captured, not yet run
        direct(c, 250.0)
        replay()                                            # another eps's table before it
        direct(c, 250.0)                                    # the graph's table before it
        replay()
        direct(c, 100.0)
        direct(c, 100.0)
        replay()
        c.close()

"""HostPipeline: steps from pinned host buffers with the copies overlapped with
compute must give, step by step, exactly the outputs of the plain in-order
StepRunner on the same inputs (the pipeline only reorders copies, never compute).
"""
import pytest
import torch

import workloads
from gpu_helpers import problem_of, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import __graft_entry__
    __graft_entry__.build()


def test_pipeline_matches_in_order_steps():
    import paper_2608_16188_gb300 as vm
    cfg = workloads.Config("pipe", 70, T=3, N=197, d=256, f=512, E=4, k=2, cf=1.25, dtype="bf16",
                           bias="drift")
    inp = to_dev(workloads.make_inputs(cfg))
    p = problem_of(cfg)
    steps = 5
    g = torch.Generator().manual_seed(3)
    xs = [(torch.randn(inp["x"].shape, generator=g).to(torch.bfloat16).pin_memory(),
           torch.randn(inp["dy"].shape, generator=g).to(torch.bfloat16).pin_memory())
          for _ in range(steps)]
    outs = [(torch.empty(inp["x"].shape, dtype=torch.bfloat16).pin_memory(),
             torch.empty(inp["x"].shape, dtype=torch.bfloat16).pin_memory()) for _ in range(steps)]
    weights = {k: v for k, v in inp.items() if k not in ("x", "dy")}
    pipe = vm.HostPipeline(p, weights, device="cuda")
    pipe.run(xs, outs)
    torch.cuda.synchronize()
    ref = vm.StepRunner(p, dict(inp))
    for i in range(steps):
        ref.inp["x"].copy_(xs[i][0])
        ref.inp["dy"].copy_(xs[i][1])
        ref.step()
        torch.cuda.synchronize()
        assert torch.equal(outs[i][0], ref.b.y.cpu()), i
        assert torch.equal(outs[i][1], ref.b.dx.cpu()), i
    assert vm.vmoe_device_status() == 0


def test_calls_follow_the_current_stream():
    """With no stream argument a call goes to torch's current stream: work queued there before it is seen, on the
    default stream and on another one."""
    import paper_2608_16188_gb300 as vm
    p = vm.problem(1, 64, 256, 128, 4, 2, 4.0, "bf16", flags=vm.VMOE_LOGITS_IN)
    for side in (None, torch.cuda.Stream()):
        with torch.cuda.stream(side):
            assert vm._stream(None) == torch.cuda.current_stream().cuda_stream
            logits = torch.zeros(1, 64, 4, device="cuda")
            out = [torch.empty(1, 64, 2, dtype=d, device="cuda") for d in (torch.int32, torch.float32, torch.int32)]
            load = torch.empty(1, 4, dtype=torch.int32, device="cuda")
            torch.cuda._sleep(2_000_000)
            logits[..., 3] = 1.0
            vm.vmoe_route(p, None, None, None, logits, *out, load)
            assert load.tolist() == [[64, 0, 0, 64]]

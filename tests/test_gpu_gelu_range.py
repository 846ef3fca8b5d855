"""GELU' of the tensor-core epilogues where it is 0 or 1: large |h|, up to where h^2 overflows."""
import pytest
import torch

import paper_2608_16188_gb300 as vm
from test_gpu_parity import _lib  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu
D = 128


@pytest.mark.parametrize("tanh", [False, True], ids=["erf", "tanh"])
def test_derivative_far_from_zero(tanh):
    p = vm.problem(1, D, D, D, 1, 1, 1.0, "bf16", vm.VMOE_GELU_TANH if tanh else 0)
    mag = torch.logspace(1.2, 18.9, D // 2, dtype=torch.float64)  # |GELU' - step| < 1e-30 from |h| = 15.8 on
    row = torch.cat([mag, -mag]).bfloat16()
    h = row[None].repeat(D, 1)
    h[1, 0], h[2, 64] = float("nan"), float("nan")
    h = h.cuda()
    load = torch.tensor([[D]], dtype=torch.int32, device="cuda")
    eye, ones = torch.eye(D, dtype=torch.bfloat16, device="cuda"), torch.ones(D, D, dtype=torch.bfloat16, device="cuda")
    dxe, dw1, dw2 = (torch.empty(D, D, dtype=torch.bfloat16, device="cuda") for _ in range(3))
    ws = torch.empty(vm.vmoe_expert_bwd_workspace_size(p), dtype=torch.uint8, device="cuda")
    vm.vmoe_expert_bwd(p, ones, h, ones, eye, eye, ones, load, dxe, dw1, dw2, ws)
    torch.cuda.synchronize()
    dh = ws.view(torch.bfloat16).double().reshape(2, D, D).sum(0)
    nan = torch.isnan(h)
    step = (h > 0).double()
    assert torch.isnan(dh[nan]).all()
    assert ((dh - step).abs()[~nan] <= 1e-7).all(), (dh - step).abs()[~nan].max()

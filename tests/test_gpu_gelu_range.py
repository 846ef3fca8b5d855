"""GELU of the tensor-core epilogues relative to its value in the negative tail, and GELU' where it is 0 or 1: large
|h|, up to where h^2 overflows."""
import math

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


@pytest.mark.parametrize("tanh", [False, True], ids=["erf", "tanh"])
def test_gelu_relative_in_the_negative_tail(tanh):
    """Every bf16 h in [-5, -2^-8]: within half a bf16 ulp of the value (2^-8) and what the approximation adds --
    formula 7.1.26 evaluated in 64 bits is at most 1.59e-3 of the tail off down to -5; the tanh form has four
    fp32 roundings in its exponent, |2 u| <= 17 at -5, and two approximate instructions: 17 * 2^-22 + 2^-21."""
    bits = torch.arange(0x3B80, 0x40A1, dtype=torch.int32)
    v = (bits | 0x8000).to(torch.int16).view(torch.bfloat16)
    rows = -(-v.numel() // D)
    x = torch.zeros(128, D, dtype=torch.bfloat16)
    x.view(-1)[:v.numel()] = v
    assert v.double().min() == -5.0 and rows <= 128
    p = vm.problem(1, D, D, D, 1, 1, 1.0, "bf16", vm.VMOE_GELU_TANH if tanh else 0)
    load = torch.tensor([[D]], dtype=torch.int32, device="cuda")
    eye = torch.eye(D, dtype=torch.bfloat16, device="cuda")
    h, a, ye = (torch.empty(D, D, dtype=torch.bfloat16, device="cuda") for _ in range(3))
    vm.vmoe_expert_fwd(p, x.cuda(), eye, eye, load, h, a, ye)
    torch.cuda.synchronize()
    hv = v.double()
    if tanh:
        u = math.sqrt(2.0 / math.pi) * (hv + 0.044715 * hv ** 3)
        want, more = hv / (1.0 + torch.exp(-2.0 * u)), 17 * 2.0 ** -22 + 2.0 ** -21
    else:
        want, more = hv * 0.5 * torch.special.erfc(-hv / math.sqrt(2.0)), 1.6e-3
    got = a.cpu().double().view(-1)[:v.numel()]
    off = ((got - want) / want).abs()
    assert (off <= 2.0 ** -8 + more).all(), (hv[off.argmax()], off.max())

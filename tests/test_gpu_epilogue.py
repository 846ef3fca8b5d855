"""GELU and GELU' of the tensor-core epilogues over the bf16 range, value by value: with identity weights H = Xe
exactly, A = GELU(H) and dH = dYe * GELU'(H) can be read off against 64-bit values.

Bounds: the erf approximation is good to 1.5e-7 (tanh form: a few fp32 roundings), so A is within bf16's half ulp,
at most 2^-8 |A| (8 significant bits), plus 2e-7 |h|, and dH = value + residual within 2^-16 |dH| plus 1e-6 (1 + |h|) of fp32 arithmetic."""
import math

import numpy as np
import pytest
import torch

import paper_2608_16188_gb300 as vm
from test_gpu_parity import _lib  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu
D = 128


def _grid():
    """128 x 128 bf16 values: every one of magnitude 2^-15 .. 2^6, then zeros, tiny and huge ones."""
    mag = torch.arange((127 - 15) << 7, (127 + 6) << 7, dtype=torch.int32)
    v = torch.cat([mag, mag | 0x8000]).to(torch.int16).view(torch.bfloat16)
    more = torch.tensor([0.0, -0.0, 1e-38, -1e-38, 1e-30, -1e-30, 1e4, -1e4, 1e18, -1e18], dtype=torch.bfloat16)
    return torch.cat([v, more, torch.zeros(D * D - v.numel() - more.numel(), dtype=torch.bfloat16)]).reshape(D, D)


def _exact(h, tanh):
    a = math.sqrt(2.0 / math.pi)
    if tanh:
        with np.errstate(over="ignore"):
            s = 1.0 / (1.0 + np.exp(np.minimum(-2.0 * a * (h + 0.044715 * h ** 3), 700.0)))
        return h * s, s + h * s * (1 - s) * 2 * a * (1 + 3 * 0.044715 * h * h)
    Phi = 0.5 * np.array([math.erfc(-v / math.sqrt(2.0)) for v in h.ravel()]).reshape(h.shape)
    return h * Phi, Phi + h * np.exp(-0.5 * h * h) / math.sqrt(2 * math.pi)


@pytest.mark.parametrize("tanh", [False, True], ids=["erf", "tanh"])
def test_gelu_value_by_value(tanh):
    p = vm.problem(1, D, D, D, 1, 1, 1.0, "bf16", vm.VMOE_GELU_TANH if tanh else 0)
    grid = _grid()
    x, eye = grid.cuda(), torch.eye(D, dtype=torch.bfloat16, device="cuda")
    e = lambda: torch.empty(D, D, dtype=torch.bfloat16, device="cuda")  # noqa: E731
    load = torch.tensor([[D]], dtype=torch.int32, device="cuda")
    h, a, ye, dxe, dw1, dw2 = (e() for _ in range(6))
    vm.vmoe_expert_fwd(p, x, eye, eye, load, h, a, ye)
    ws = torch.empty(vm.vmoe_expert_bwd_workspace_size(p), dtype=torch.uint8, device="cuda")
    aux = grid.clone()  # H with infinities and NaN in some columns: they stay in their own elements
    aux[::2, 5], aux[1::2, 6], aux[::3, 9] = math.inf, -math.inf, math.nan
    ones = torch.ones(D, D, dtype=torch.bfloat16, device="cuda")
    vm.vmoe_expert_bwd(p, x, aux.cuda(), a, eye, eye, ones, load, dxe, dw1, dw2, ws)
    torch.cuda.synchronize()
    assert vm.vmoe_device_status() == 0
    hv = grid.double().numpy()
    assert torch.equal(h.cpu(), grid)
    ref, _ = _exact(hv, tanh)
    err = np.abs(a.double().cpu().numpy() - ref)
    bad = err > 2.0 ** -8 * 1.001 * np.abs(ref) + 2e-7 * np.abs(hv) + 1e-40
    assert not bad.any(), (hv[bad][:8], err[bad][:8])
    fine = torch.isfinite(aux).numpy()
    av = np.where(fine, aux.double().numpy(), 0.0)
    dh = ws.view(torch.bfloat16).double().cpu().numpy().reshape(2, D, D)
    _, dref = _exact(av, tanh)
    small = fine & (np.abs(av) < 1e3)  # beyond, (1 - s) s and exp(-h^2 / 2) are 0 and GELU' is 0 or 1
    derr = np.abs(dh[0] + dh[1] - dref)
    bad = small & (derr > 2.0 ** -16 * np.abs(dref) + 1e-6 * (1 + np.abs(av)))
    assert not bad.any(), (av[bad][:8], derr[bad][:8])
    assert np.all(np.isfinite(dh[0])[fine]) and np.all(np.isnan(dh[0])[torch.isnan(aux).numpy()])

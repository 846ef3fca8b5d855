"""The attention core at every edge of its blocks: groups whose loads sit at and beside multiples of 16, 32, 64 and 128,
in the fused backward of 128 and of 256 rows and in the two kernels above, with NaN in every padding row.  O and
dQ|dK|dV against 64 bits from the Q, K, V, O and dO that the core received, to the bars of the parity tests (2e-2 of
an output's RMS an element, 5e-3 in all)."""
import numpy as np
import pytest
import torch

import paper_2608_16188_gb300 as vm
from gpu_helpers import BF16_RMS_TOL, BF16_TOL, rel_err, rms_err
from test_gpu_parity import _lib  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu
H, HD, D = 2, 128, 128


@pytest.mark.parametrize("C", [128, 256, 330])
def test_core_at_block_edges(C):
    at = sorted({v for m in (16, 32, 48, 64, 96, 128, 160, 192, 224, 256, 320) for v in (m - 1, m, m + 1) if v <= C} | {0, 1, C})
    E = len(at)
    p = vm.problem(1, C, D, 128, E, 1, 1.0, "bf16", capacity=C)
    g = torch.Generator(device="cuda").manual_seed(C)
    r = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    load = torch.tensor([at], dtype=torch.int32, device="cuda")
    pad = torch.arange(C, device="cuda")[None, :] >= load[0][:, None]
    nan = lambda *s, dt=torch.bfloat16: torch.full(s, float("nan"), dtype=dt, device="cuda")  # noqa: E731
    xe, dye = r(E, C, D).bfloat16(), r(E, C, D).bfloat16()
    xe[pad], dye[pad] = float("nan"), float("nan")
    wqkv, wo = (r(E, D, 3 * HD) / D ** 0.5).bfloat16(), (r(E, HD, D) / HD ** 0.5).bfloat16()
    qkv, o, ye, lse = nan(E, C, 3 * HD), nan(E, C, HD), nan(E, C, D), nan(E, H, C, dt=torch.float32)
    dxe, dwqkv, dwo = nan(E, C, D), nan(E, D, 3 * HD), nan(E, HD, D)
    ws = nan(vm.vmoe_attn_expert_bwd_workspace_size(p, H) // 2)
    vm.vmoe_attn_expert_fwd(p, H, xe, wqkv, wo, load, qkv, o, lse, ye)
    vm.vmoe_attn_expert_bwd(p, H, xe, qkv, o, lse, wqkv, wo, dye, load, dxe, dwqkv, dwo, ws)
    torch.cuda.synchronize()
    assert vm.vmoe_device_status() == 0
    dout, dqkv = ws[:E * C * HD].view(E, C, HD), ws[E * C * HD:E * C * HD * 4].view(E, C, 3 * HD)
    for e, L in enumerate(at):
        if L == 0:
            assert not dwqkv[e].any() and not dwo[e].any()
            continue
        heads = lambda t: t[e, :L].double().reshape(L, -1, 64).transpose(0, 1)  # noqa: E731
        q, k, v = heads(qkv).split(H)
        do, ob = heads(dout), heads(o)
        P = torch.softmax(q @ k.transpose(1, 2) / 8, dim=2)
        dS = P * (do @ v.transpose(1, 2) - (do * ob).sum(2, keepdim=True)) / 8
        ref = {"o": (ob, P @ v), "dq": (heads(dqkv)[:H], dS @ k), "dk": (heads(dqkv)[H:2 * H], dS.transpose(1, 2) @ q),
               "dv": (heads(dqkv)[2 * H:], P.transpose(1, 2) @ do)}
        for n, (got, want) in ref.items():
            want = want.cpu().numpy()
            if not np.abs(want).max() > 1e-12:  # one token: dQ and dK are zero but for the rounding of O
                continue
            if L == 1 and n in ("dq", "dk"):  # P = 1 and dP - D is O's rounding error alone
                assert float((got.cpu() - torch.from_numpy(want)).abs().max()) < 1e-2
                continue
            assert rel_err(got, want) <= BF16_TOL and rms_err(got, want) <= BF16_RMS_TOL, (L, n, rel_err(got, want))
        assert torch.isfinite(ye[e, :L]).all() and torch.isfinite(dxe[e, :L]).all()
    assert torch.isnan(qkv[pad]).all() and torch.isnan(o[pad]).all() and torch.isnan(dqkv[pad]).all()
    assert torch.isfinite(dwqkv).all() and torch.isfinite(dwo).all()

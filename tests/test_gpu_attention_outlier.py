"""One query row that is huge, infinite or NaN, in groups above 128 tokens: dQ of every other row stays bit for bit
what it is without it (dK and dV sum over the queries, so they see it)."""
import pytest
import torch

import paper_2608_16188_gb300 as vm
from test_gpu_parity import _lib  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu
T, E, D, H = 1, 6, 256, 4


@pytest.mark.parametrize("C", [129, 200, 256, 330])
@pytest.mark.parametrize("what", ["huge dY", "inf dY", "nan dY", "huge Q", "nan Q"])
def test_other_rows_keep_their_dq(C, what):
    gen = torch.Generator(device="cuda").manual_seed(C)
    r = lambda *s, k=1.0: (torch.randn(s, generator=gen, device="cuda") * k).bfloat16()  # noqa: E731
    e = lambda *s, dt=torch.bfloat16: torch.empty(s, device="cuda", dtype=dt)  # noqa: E731
    p = vm.problem(T, 2 * C, D, D, E, 1, 1.0, capacity=C)
    load = torch.tensor([[C, C - 1, 65, 33, 17, 2]], dtype=torch.int32, device="cuda")
    xe, dye = r(T, E, C, D), r(T, E, C, D)
    wqkv, wo = r(T, E, D, 192 * H, k=D ** -0.5), r(T, E, 64 * H, D, k=(64 * H) ** -0.5)
    qkv, o, lse, ye = e(T, E, C, 192 * H), e(T, E, C, 64 * H), e(T, E, H, C, dt=torch.float32), e(T, E, C, D)
    vm.vmoe_attn_expert_fwd(p, H, xe, wqkv, wo, load, qkv, o, lse, ye)
    dxe, dwqkv, dwo = torch.zeros_like(xe), torch.empty_like(wqkv), torch.empty_like(wo)
    ws = e(vm.vmoe_attn_expert_bwd_workspace_size(p, H), dt=torch.uint8)
    row, rows, hd = 1, T * E * C, 64 * H

    def dq(dy, q):
        vm.vmoe_attn_expert_bwd(p, H, xe, q, o, lse, wqkv, wo, dy, load, dxe, dwqkv, dwo, ws)
        torch.cuda.synchronize()
        return ws[rows * hd * 2:rows * hd * 8].view(torch.bfloat16).reshape(E, C, 3 * hd)[..., :hd].clone()

    ref = dq(dye, qkv)
    dy, q = dye.clone(), qkv.clone()
    value = {"huge": 2.0 ** 40, "inf": float("inf"), "nan": float("nan")}[what.split()[0]]
    if what.endswith("Q"):
        q[:, :, row, :hd] = q[:, :, row, :hd] * value
    else:
        dy[:, :, row] = dy[:, :, row] * value
    got = dq(dy, q)
    assert vm.vmoe_device_status() == 0
    for g, n in enumerate(load[0].tolist()):
        keep = [i for i in range(n) if i != row]
        assert torch.isfinite(ref[g, keep]).all()
        assert torch.equal(got[g, keep], ref[g, keep]), (g, n)

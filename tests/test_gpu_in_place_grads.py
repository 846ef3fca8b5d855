"""Gradients stored over the weights that an earlier launch of the same call reads (a caller
short of memory): bit for bit what separate buffers get."""
import pytest
import torch

import paper_2608_16188_gb300 as vm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _randn(gen, *shape, scale=1.0):
    return (torch.randn(shape, generator=gen, device="cuda") * scale).bfloat16()


@pytest.mark.parametrize("d,f,C,budget", [(256, 512, 100, 1.0), (384, 1152, 300, 1.0), (256, 512, 100, 0.3)])
def test_ffn_gradients_over_the_weights(d, f, C, budget):
    T, E = 3, 16
    gen = torch.Generator(device="cuda").manual_seed(d + C)
    p = vm.problem(T, 4 * C, d, f, E, 2, 1.0, capacity=C)
    load = torch.randint(0, C + 1, (T, E), generator=gen, device="cuda", dtype=torch.int32)
    load[0, 0], load[0, 1], load[1, 0] = 0, C, 1
    xe, dye = _randn(gen, T, E, C, d), _randn(gen, T, E, C, d)
    w1, w2 = _randn(gen, T, E, d, f, scale=d ** -0.5), _randn(gen, T, E, f, d, scale=f ** -0.5)
    h, a = torch.empty(2, T, E, C, f, device="cuda", dtype=torch.bfloat16)
    ye = torch.empty_like(xe)
    vm.vmoe_expert_fwd(p, xe, w1, w2, load, h, a, ye)
    size = max(vm.vmoe_expert_bwd_min_workspace_size(p), int(vm.vmoe_expert_bwd_workspace_size(p) * budget))
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")

    def run(in_place):
        v1, v2 = w1.clone(), w2.clone()
        g1, g2 = (v1, v2) if in_place else (torch.empty_like(v1), torch.empty_like(v2))
        dxe = torch.zeros_like(xe)
        # dW2 of a call in slices comes before dA, which reads W2
        vm.vmoe_expert_bwd(p, xe, h, a, v1, v2, dye, load, dxe, g1, g2 if budget == 1.0 else torch.empty_like(v2), ws)
        return dxe, g1, g2 if budget == 1.0 else g1

    want = run(False)
    for _ in range(20):
        for got, ref in zip(run(True), want):
            assert torch.equal(got, ref)
    assert vm.vmoe_device_status() == 0


@pytest.mark.parametrize("C", [100, 200])
def test_attention_gradients_over_the_weights(C):
    T, E, d, H = 2, 16, 256, 4
    gen = torch.Generator(device="cuda").manual_seed(C)
    p = vm.problem(T, 4 * C, d, d, E, 2, 1.0, capacity=C)
    load = torch.randint(0, C + 1, (T, E), generator=gen, device="cuda", dtype=torch.int32)
    e = lambda *s, dtype=torch.bfloat16: torch.empty(s, device="cuda", dtype=dtype)  # noqa: E731
    xe, dye = _randn(gen, T, E, C, d), _randn(gen, T, E, C, d)
    wqkv, wo = _randn(gen, T, E, d, 192 * H, scale=d ** -0.5), _randn(gen, T, E, 64 * H, d, scale=(64 * H) ** -0.5)
    qkv, o, lse, ye = e(T, E, C, 192 * H), e(T, E, C, 64 * H), e(T, E, H, C, dtype=torch.float32), e(T, E, C, d)
    vm.vmoe_attn_expert_fwd(p, H, xe, wqkv, wo, load, qkv, o, lse, ye)
    ws = e(vm.vmoe_attn_expert_bwd_workspace_size(p, H), dtype=torch.uint8)

    def run(in_place):
        a, b = wqkv.clone(), wo.clone()
        ga, gb = (a, b) if in_place else (torch.empty_like(a), torch.empty_like(b))
        dxe = torch.zeros_like(xe)
        vm.vmoe_attn_expert_bwd(p, H, xe, qkv, o, lse, a, b, dye, load, dxe, ga, gb, ws)
        return dxe, ga, gb

    want = run(False)
    for _ in range(20):
        for got, ref in zip(run(True), want):
            assert torch.equal(got, ref)
    assert vm.vmoe_device_status() == 0

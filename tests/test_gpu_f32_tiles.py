"""fp32 groups that hold far fewer rows than their capacity: a capacity of 33 costs about what 32 costs (tiles of
64 rows against tiles of 32), many groups or not.  Times are the kernel trace's, the fastest of 20 launches; the
factor of two allowed is below the 2.7 that 128-row tiles took and above the 0.9 to 1.4 of 64-row ones."""
import pytest
import torch

import paper_2608_16188_gb300 as vm
from test_gpu_parity import _lib  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu


def _times(C, L, T=8, E=64, d=64, f=256):
    p = vm.problem(T, 64, d, f, E, 2, 1.0, "f32", capacity=C)
    gen = torch.Generator(device="cuda").manual_seed(C)
    r = lambda *s: torch.randn(s, generator=gen, device="cuda")  # noqa: E731
    load = torch.full((T, E), L, dtype=torch.int32, device="cuda")
    xe, dye, w1, w2 = r(T, E, C, d), r(T, E, C, d), r(T, E, d, f), r(T, E, f, d)
    h, a = torch.empty(2, T, E, C, f, device="cuda")
    ye, dxe, dw1, dw2 = (torch.empty_like(t) for t in (xe, xe, w1, w2))
    ws = torch.empty(T * E * C * f, device="cuda")
    vm.vmoe_trace_enable(6 * 20)
    for _ in range(20):
        vm.vmoe_expert_fwd(p, xe, w1, w2, load, h, a, ye)
        vm.vmoe_expert_bwd(p, xe, h, a, w1, w2, dye, load, dxe, dw1, dw2, ws)
    torch.cuda.synchronize()
    best = {}
    for i in range(vm.vmoe_trace_disable()):
        name, ms = vm.vmoe_trace_get(i)
        best[name] = min(ms, best.get(name, ms))
    want = torch.nn.functional.gelu(xe[:, :, :L].double() @ w1.double()) @ w2.double()
    got = ye[:, :, :L].double()
    assert ((got - want).norm() / want.norm()) < 1e-5
    return best


def test_capacity_33_costs_what_32_does():
    a, b = _times(32, 10), _times(33, 10)
    assert set(a) == set(b) and len(a) == 6
    for n in a:
        assert b[n] < 2.0 * a[n], (n, a[n], b[n])

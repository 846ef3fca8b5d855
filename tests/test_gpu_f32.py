"""fp32 problems where the CUDA-core kernels change path: row tiles of 16, 32 and 64 with ragged edges, K ranges
split over a cluster, router chunks and expert passes with remainders, one token.  Held to the fp32 bars of the
parity tests (1e-5 of an output's RMS: sums of a few hundred to a few thousand fp32 products in any order stay
under 1e-6)."""
import pytest

import workloads
from gpu_helpers import run_step, to_dev
from test_gpu_parity import _compare_step, _lib  # noqa: F401  (the fixture that builds the library)

pytestmark = pytest.mark.gpu

Config = workloads.Config
CASES = [
    # 64 groups: no K split; d = 72 and f = 1028 end inside a tile and a K chunk
    Config("f32_wide_tiles", 90, T=2, N=300, d=72, f=1028, E=32, k=2, cf=1.25, dtype="f32", bias="drift"),
    # 2 groups, K = 516 (33 chunks) over 8 CTAs; row tiles of 64 and of 2 rows
    Config("f32_split", 91, T=1, N=66, d=128, f=516, E=2, k=2, cf=1.0, dtype="f32", flags=4),
    # 70 experts (two router passes of 64), d = 136 (a chunk of 8), empty groups
    Config("f32_experts70", 92, T=2, N=45, d=136, f=64, E=70, k=3, cf=1.0, dtype="f32", bias="zipf", flags=2),
    # 13 and 27 rows a group: tiles of 16 and 32 rows, d and f off the 128-wide columns, with and without a split
    Config("f32_rows13", 89, T=3, N=124, d=136, f=428, E=30, k=2, cf=1.5, dtype="f32", bias="drift"),
    Config("f32_rows27", 88, T=1, N=50, d=200, f=260, E=4, k=1, cf=2.1, dtype="f32"),
    Config("f32_one_token", 93, T=1, N=1, d=8, f=4, E=2, k=1, cf=1.0, dtype="f32"),
]


@pytest.mark.parametrize("cfg", CASES, ids=lambda c: c.name)
def test_f32_step_parity(cfg):
    inp = workloads.make_inputs(cfg)
    _, b = run_step(cfg, to_dev(inp))
    _compare_step(cfg, inp, b, cfg.flags)


@pytest.mark.parametrize("N,d,E", [(1, 8, 3), (300, 72, 70), (1100, 40, 13), (257, 136, 64)])
def test_f32_router_dw_splits(N, d, E):
    """dW_r and dbias of fp32 problems, the tokens over one to eight CTAs with remainders in tokens, d and experts:
    fp32 sums of up to 1100 products in two levels stay under 1e-6 of 64 bits."""
    import torch

    import paper_2608_16188_gb300 as vm
    T, k = 2, 2
    p = vm.problem(T, N, d, 4, E, k, 2.0, "f32", capacity=N)
    g = torch.Generator(device="cuda").manual_seed(N)
    r = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    e = lambda *s, dt=torch.float32: torch.empty(s, dtype=dt, device="cuda")  # noqa: E731
    x, wr, dy, ye = r(T, N, d), r(T, d, E) / d ** 0.5, r(T, N, d), r(T, E, N, d)
    logits, gate, idx, slot = e(T, N, E), e(T, N, k), e(T, N, k, dt=torch.int32), e(T, N, k, dt=torch.int32)
    vm.vmoe_route(p, x, wr, None, logits, idx, gate, slot, e(T, E, dt=torch.int32))
    dgate, dl, dw, db = e(T, N, k), e(T, N, E), e(T, d, E), e(T, E)
    vm.vmoe_router_bwd(p, x, wr, logits, idx, gate, slot, dy, ye, dgate, dl, dw, db, None)
    ref = x.double().transpose(1, 2) @ dl.double()
    assert float((dw - ref).norm() / ref.norm()) < 1e-6
    rb = dl.double().sum(1)
    assert float((db - rb).abs().max()) < 1e-5 * float(dl.abs().sum(1).max())

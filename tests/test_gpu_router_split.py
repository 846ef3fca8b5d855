"""The bf16 router where a cluster of CTAs shares a token tile: chunks of d with remainders, more splits than a power of
two, two passes of experts, ragged tokens.  Logits to 1e-5 of the 64-bit ones (fp32 sums of up to 1024 exact products
stay under 3e-6), choices and slots exactly those of the GPU's own logits, gates to 1e-6."""
import numpy as np
import pytest
import torch

import oracle
import paper_2608_16188_gb300 as vm
import workloads
from gpu_helpers import GATE_RTOL, np64, problem_of, rel_err, to_dev
from test_gpu_parity import _lib  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu

Config = workloads.Config
CASES = [
    Config("split_6", 95, T=4, N=197, d=768, f=128, E=32, k=2, cf=1.25, dtype="bf16", bias="drift"),  # 6 CTAs a tile
    Config("split_8_e70", 96, T=1, N=130, d=1024, f=128, E=70, k=3, cf=1.0, dtype="bf16"),  # 8 CTAs, two passes
    Config("split_5_tail", 97, T=2, N=65, d=520, f=128, E=5, k=2, cf=1.0, dtype="bf16", flags=2),  # a chunk of 8
    Config("no_split_tail", 94, T=2, N=65, d=136, f=128, E=5, k=2, cf=1.0, dtype="bf16", flags=2),
    Config("split_7", 98, T=1, N=1, d=840, f=128, E=33, k=8, cf=8.0, dtype="bf16"),  # 7 CTAs, one token, top-8
    Config("no_split", 99, T=3, N=3300, d=264, f=128, E=40, k=1, cf=1.0, dtype="bf16", bias="zipf"),  # one CTA a tile
]


@pytest.mark.parametrize("cfg", CASES, ids=lambda c: c.name)
def test_route(cfg):
    inp = workloads.make_inputs(cfg, with_weights=False)
    dev = to_dev(inp)
    p = problem_of(cfg)
    C = vm.vmoe_problem_capacity(p)
    e = lambda *s, dtype=torch.int32: torch.empty(s, dtype=dtype, device="cuda")  # noqa: E731
    logits, gate = e(cfg.T, cfg.N, cfg.E, dtype=torch.float32), e(cfg.T, cfg.N, cfg.k, dtype=torch.float32)
    idx, slot, load = e(cfg.T, cfg.N, cfg.k), e(cfg.T, cfg.N, cfg.k), e(cfg.T, cfg.E)
    vm.vmoe_route(p, dev["x"], dev["w_router"], dev["bias"], logits, idx, gate, slot, load)
    torch.cuda.synchronize()
    ref = np.einsum("tnd,tde->tne", np64(inp["x"]), np64(inp["w_router"]))
    if inp["bias"] is not None:
        ref = ref + np64(inp["bias"])[:, None]
    assert rel_err(logits, ref) < 1e-5
    ridx, rgate, rslot, rload = oracle.route(logits.cpu().numpy(), cfg.k, C, cfg.flags)
    assert np.array_equal(idx.cpu().numpy(), ridx)
    assert np.array_equal(slot.cpu().numpy(), rslot)
    assert np.array_equal(load.cpu().numpy(), rload)
    np.testing.assert_allclose(gate.cpu().numpy(), rgate, rtol=GATE_RTOL)


def test_ties_and_minus_infinity_by_warp():
    """Equal logits and -inf biases through the warp's choice: lowest index first, indices in range."""
    T, N, d, E, k = 1, 40, 256, 40, 5
    x = torch.zeros(T, N, d, dtype=torch.bfloat16, device="cuda")
    wr = torch.zeros(T, d, E, device="cuda")
    bias = torch.full((T, E), -float("inf"), device="cuda")
    bias[0, [3, 35, 7]] = 1.0
    p = vm.problem(T, N, d, 128, E, k, 40.0)
    e = lambda *s, dtype=torch.int32: torch.empty(s, dtype=dtype, device="cuda")  # noqa: E731
    logits, idx, gate = e(T, N, E, dtype=torch.float32), e(T, N, k), e(T, N, k, dtype=torch.float32)
    vm.vmoe_route(p, x, wr, bias, logits, idx, gate, e(T, N, k), e(T, E))
    assert idx[0].cpu().tolist() == [[3, 7, 35, 0, 1]] * N
    assert torch.allclose(gate[0].cpu(), torch.tensor([1 / 3, 1 / 3, 1 / 3, 0.0, 0.0]).expand(N, k))

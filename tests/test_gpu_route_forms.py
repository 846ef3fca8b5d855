"""The fp32 router's form for many tokens (64 a CTA, chunks of 32) at the edges of its rule and its tiles, and the
capacity scan's ways from ranks to slots: with few and with many counters, choices apart in memory, and with the
indices in shared memory or not.  Held as in test_gpu_router_split: logits to 1e-5 of 64 bits (sums of up to 520 fp32
products in any order stay under 1e-6), choices, slots and loads exactly those of the GPU's own logits."""
import pytest

import test_gpu_router_split as split
import workloads
from test_gpu_parity import _lib  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu

Config = workloads.Config


def _c(name, seed, dtype="f32", **kw):
    return Config(name, seed, **dict(dict(f=4 if dtype == "f32" else 128, k=2, cf=1.0, dtype=dtype), **kw))


CASES = [
    _c("many_e12_d8", 201, T=16, N=640, d=8, E=12, k=4),          # whole tiles, a chunk of 8
    _c("many_e32_d520", 202, T=3, N=3300, d=520, E=32),           # 36 tokens in the last tile
    _c("many_e33_d136", 203, T=8, N=1300, d=136, E=33, k=1, bias="zipf"),  # the 64-expert pass, half empty
    _c("many_e60_top8", 204, T=17, N=577, d=40, E=60, k=8, flags=2),
    _c("many_e200", 205, T=5, N=2000, d=24, E=200, k=3),          # four passes of experts
    _c("half_d512", 206, T=1, N=5000, d=512, E=16),               # 79 tiles: many up to d 512 ...
    _c("half_d520", 207, T=1, N=5000, d=520, E=16),               # ... and few beyond
    _c("scan_e128", 208, "bf16", T=2, N=90, d=128, E=128, k=4),
    _c("scan_e129", 209, "bf16", T=1, N=11, d=128, E=129, k=8),
    _c("scan_e256", 210, "bf16", T=4, N=70, d=128, E=256, k=2),
    _c("scan_top3", 211, "bf16", T=1, N=33, d=128, E=7, k=3, cf=0.4),
    _c("scan_top8_shared", 212, "bf16", T=2, N=1500, d=128, E=9, k=8, cf=0.7),
    _c("scan_top8_global", 213, "bf16", T=2, N=1700, d=128, E=9, k=8, cf=0.7),
    _c("scan_one_token", 214, "bf16", T=3, N=1, d=128, E=31, k=4, cf=9.0),
]


@pytest.mark.parametrize("cfg", CASES, ids=lambda c: c.name)
def test_route(cfg):
    split.test_route(cfg)

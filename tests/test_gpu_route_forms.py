"""The capacity scan's ways from ranks to slots: with few and with many counters, choices apart in memory, and with the
indices in shared memory or not.  Held as in test_gpu_router_split: choices, slots and loads exactly those of the
GPU's own logits."""
import pytest

import test_gpu_router_split as split
import workloads
from test_gpu_parity import _lib  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu

Config = workloads.Config


def _c(name, seed, dtype="f32", **kw):
    return Config(name, seed, **dict(dict(f=4 if dtype == "f32" else 128, k=2, cf=1.0, dtype=dtype), **kw))


CASES = [
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

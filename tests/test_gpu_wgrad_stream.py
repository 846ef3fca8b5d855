"""The SM-pair weight gradients with nothing resident: more than 256 rows a group, M and N ending in half a 256-wide
tile, empty groups, more tiles than pairs (so that pairs take further ones), every residue of the last k-block -- held,
like every tail, to the bars of test_gpu_tails and to bitwise equality with the sliced backward."""
import numpy as np
import pytest

from test_gpu_tails import _check_tails, _lib  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,f,C,loads", [
    (256, 512, 330, [0, 1, 15, 16, 17, 63, 64, 65, 255, 256, 257, 271, 272, 320, 321, 329, 330]),
    (384, 640, 128, [0, 1, 16, 31, 63, 64, 65, 96, 127, 128, 0, 50]),
    (640, 384, 40, [0, 40, 39, 33, 32, 17, 16, 1, 0, 8]),
    (256, 256, 64, [int(v) for v in np.random.default_rng(5).integers(0, 65, size=200)]),  # dW2 alone streams
    (384, 384, 300, [0] + [int(v) for v in np.random.default_rng(6).integers(0, 301, size=60)]),
], ids=lambda v: str(v) if not isinstance(v, list) else "%dgroups" % len(v))
def test_streamed_tails(d, f, C, loads):
    loads = [0] + loads[1:]  # group 0 empty: its gradients must be zeros
    _check_tails("bf16", d, f, C, loads)

"""Row GEMMs in 192-column tiles (plain stores, N a multiple of 192 but not of 256, at most 128 rows a group): partial
and full row tiles, empty groups, SMs that take one tile and several, two and six tiles across -- held to the bars of
test_gpu_tails and to bitwise equality with the sliced backward, whose slices take other widths."""
import numpy as np
import pytest

from test_gpu_tails import LOADS, _check_tails, _lib  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,f,loads", [
    (384, 256, LOADS * 3),  # 132 tiles instead of 198
    (1152, 128, LOADS[:20]),  # 120 instead of 180
    (384, 512, [int(v) for v in np.random.default_rng(8).integers(0, 129, size=150)]),  # 300 instead of 450
], ids=lambda v: str(v) if not isinstance(v, list) else "%dgroups" % len(v))
def test_row_tiles_of_192(d, f, loads):
    _check_tails("bf16", d, f, 128, [0] + loads[1:])

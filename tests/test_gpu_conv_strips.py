"""Strip lengths of the convolution: shortest strips (16 rows) with a remainder, lengths between the limits, full ones."""
import pytest

from test_gpu_conv import TOL, _run
from workloads import make_forest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 16, 17, 4737, 9500, 38001])
def test_strip_lengths(rows):
    tree = ([-1], [0], [rows]) if rows < 100 else ([-1, 0, 0, 1], [0, rows // 4, 100, 7], [rows // 2, 50, rows // 4, rows - rows // 2 - rows // 4 - 50])
    ey, ex, ew = _run(make_forest([tree]), 2048, 4, "bf16", rows)
    assert ey <= TOL["bf16"] and ex <= TOL["bf16"] and ew <= 1e-4, (ey, ex, ew)

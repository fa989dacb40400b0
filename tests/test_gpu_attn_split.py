"""The cut dK / dV work of small attention problems: key tiles whose query tiles end at and around a unit's edges, one query
head and grouped heads, and a dq tensor too small for any partial sum."""
import pytest

from test_gpu_attn import _check_backward
from workloads import make_forest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("root,kids", [(40, ()), (1024, ()), (1025, (64, 65)), (500, (1, 63, 129, 300)), (600, (130,) * 6)])
@pytest.mark.parametrize("Hq,Hkv", [(1, 1), (6, 2)])
def test_split_backward(root, kids, Hq, Hkv):
    n = len(kids)
    fo = make_forest([([-1] + [i // 2 for i in range(n)], [0] + [max(1, (root, *kids)[i // 2] - i) for i in range(n)], [root, *kids])])
    _check_backward(fo, Hq, Hkv, 7)

"""Sums over hierarchies whose first level has many groups, bit for bit against
the step executor (a traced communicator runs its schedule step by step)."""
import pytest

from tests.test_gpu_sweep import _both

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


# 32 sections, one more, the most (128) and one more, which goes to one warp;
# whole vectors and element tails
@pytest.mark.parametrize("dtype,d", [("f32", 5), ("f32", 64), ("bf16", 33), ("fp8", 128)])
@pytest.mark.parametrize("P,h", [(64, [32, 2]), (66, [33, 2]), (512, [64, 8]), (1024, [128, 8]), (258, [129, 2]),
                                 (256, [2, 32, 4])])
def test_sums_of_many_groups(P, h, dtype, d):
    _both("reduce", P, h, 1, 1, d, dtype, seed=P)

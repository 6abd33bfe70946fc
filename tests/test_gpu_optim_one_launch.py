"""The factored optimiser step in one launch, at the shapes that decide how its warps and clusters share a matrix: rows of one column
vector, rows side by side in a warp, strips with idle lanes, more strips than warps, slabs of unequal height, one to eight
blocks per matrix, and matrices on both sides of the size up to which it is taken."""
import pytest

from helpers import small_workload
from test_gpu_optim import test_factored_adam_steps as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,h,act", [(3, 8, 8, "bf16"),        # one vector a row, 32 rows side by side
                                       (40, 16, 24, "bf16"),     # two and three vectors
                                       (2, 328, 264, "bf16"),    # 41 and 33 vectors: two strips, one of them nearly idle
                                       (2, 2056, 128, "bf16"),   # 257 rows a block; 257 vectors: nine strips, one row share
                                       (2, 5000, 72, "bf16"),    # 625 vectors: more strips than warps
                                       (3, 1000, 1024, "bf16"),  # 125 rows a block
                                       (2, 1024, 2048, "bf16"),  # 4 MiB
                                       (2, 1032, 2048, "bf16"),  # more
                                       (5, 4, 260, "f32"),       # one vector a row; 65
                                       (2, 516, 1028, "f32")])  # 65 rows a block, the last one 61
def test_factored_adam_of_any_shape(n, d, h, act):
    check(small_workload(f"adam-shape-{d}-{h}", T=8, d=d, h=h, n=n, k=1, act=act, seed=69))

"""The factored optimiser step at the widths and expert counts that decide how its update walks a matrix: column vectors on whole,
partly idle and several passes of 256 threads, 16 and 64 rows a block."""
import pytest

from helpers import small_workload
from test_gpu_optim import test_factored_adam_steps as check

pytestmark = pytest.mark.gpu


# vectors of a row: bf16 width / 8, f32 width / 4
@pytest.mark.parametrize("n,d,h,act", [(2, 1088, 2056, "bf16"),  # 136 and 257 vectors: flat
                                       (1, 1784, 1792, "bf16"),  # 223 (flat) and 224 (columns)
                                       (3, 344, 4104, "bf16"),   # 43 vectors in five groups (flat), 513
                                       (600, 8, 72, "bf16"),     # 1 and 9 vectors, 64 rows a block
                                       (600, 76, 4, "f32"),      # 19 and 1 vectors
                                       (2, 1032, 1024, "f32"),   # 258 (flat) and 256 (columns, 16 rows a block)
                                       (300, 132, 68, "f32")])   # 33 and 17 vectors
def test_factored_adam_of_any_width(n, d, h, act):
    check(small_workload(f"adam-width-{d}-{h}", T=8, d=d, h=h, n=n, k=1, act=act, seed=68))

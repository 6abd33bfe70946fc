"""The projection, onto gate widths of whole quads and of single floats: every tile it is cut into, a row, a column and a feature short of and behind their borders, batches
of one row, features that fill no K block. Logits bit for bit as the oracle's chains."""
import pytest

from helpers import small_workload
from test_gpu_projection_widths import check

pytestmark = pytest.mark.gpu

# [W_g | W_noise] has 2 n columns; by the estimate of pick_tile: 16 x 16, 64 x 16, 128 x 16, 32 x 32, 64 x 64 and 64 x 128 tiles
FLAT = [(1, 4, 2, 8, "bf16"), (17, 12, 3, 72, "f32"), (300, 64, 2, 200, "bf16"), (15 * 64 + 1, 8, 1, 40, "f32"), (3001, 20, 3, 136, "bf16"),
        (20001, 4, 2, 24, "f32"), (18945, 8, 2, 104, "bf16"), (4097, 36, 4, 136, "f32"), (8193, 32, 2, 264, "bf16"), (20000, 100, 2, 72, "bf16"),
        (12001, 132, 2, 40, "f32"), (6001, 300, 4, 8, "bf16"),
        (1, 1, 1, 8, "bf16"), (17, 13, 3, 72, "f32"), (300, 65, 2, 200, "bf16"), (15 * 64 + 1, 7, 1, 40, "f32"), (3001, 21, 3, 136, "bf16"),
        (20001, 5, 2, 24, "f32"), (18945, 6, 2, 104, "bf16"), (4097, 37, 4, 136, "f32"), (8193, 47, 2, 264, "bf16"), (20000, 99, 2, 72, "bf16"),
        (6001, 301, 4, 8, "bf16"), (1025, 257, 2, 520, "bf16"), (9000, 511, 2, 40, "bf16")]


@pytest.mark.parametrize("T,n,k,d,act", FLAT)
def test_flat_logits(T, n, k, d, act):
    check(small_workload(f"tile-{T}-{n}", T=T, d=d, h=16, n=n, k=k, act=act, seed=50 + k))


@pytest.mark.parametrize("T,a,b,d,act", [(129, 4, 8, 40, "f32"), (5000, 16, 16, 72, "bf16"), (9000, 4, 64, 24, "f32"), (40, 32, 4, 8, "bf16"),
                                         (129, 5, 7, 40, "f32"), (5000, 17, 13, 72, "bf16"), (9000, 3, 66, 24, "f32"), (40, 33, 2, 8, "bf16")])
def test_grouped_logits(T, a, b, d, act):
    check(small_workload(f"tile-{a}x{b}", T=T, d=d, h=16, n=a * b, k=2, act=act, a=a, k1=2, b=b, k2=1, seed=56))


# single floats of the weights: where 128 x 64 tiles of the float product are the fewer waves, and just not
@pytest.mark.parametrize("T,n,k,d,act", [(17365, 73, 2, 72, "f32"), (11001, 75, 2, 296, "bf16"), (7117, 131, 2, 40, "f32"), (3554, 301, 2, 136, "bf16"), (4000, 93, 2, 136, "f32")])
def test_flat_logits_by_the_float_product(T, n, k, d, act):
    check(small_workload(f"tile-{T}-{n}", T=T, d=d, h=16, n=n, k=k, act=act, seed=60 + k))


# fewer rows and features than a tile has, in many columns
@pytest.mark.parametrize("T,n,k,d,act", [(3, 700, 2, 128, "f32"), (29, 724, 2, 56, "f32"), (29, 201, 2, 56, "bf16"), (5, 90, 2, 8, "bf16"), (65, 500, 2, 40, "bf16"), (1, 333, 2, 4, "f32")])
def test_few_rows_onto_many_columns(T, n, k, d, act):
    check(small_workload(f"tile-{T}-{n}-{d}", T=T, d=d, h=16, n=n, k=k, act=act, seed=70 + k))

"""The gates' gradient products of narrow gates, at the borders of their tiles, slices and rules: whole fused steps against the oracle at the
tolerances of the float paths."""
import pytest

from helpers import small_workload
from test_gpu_fused import oracle_cached, test_fused_forward_backward as check_flat
from test_gpu_hier import test_hier_fused as check_hier

pytestmark = pytest.mark.gpu

# dX: 16 x 16 tiles below 512 tokens, 32 x 32 and 64 x 64 up to 40 logits; dW: 16 logits and fewer, few blocks, up to 72 logits
FLAT = [
    small_workload("gp-one-token", T=1, d=64, h=64, n=4, k=1, seed=101),
    small_workload("gp-511", T=511, d=72, h=64, n=20, k=2, act="bf16", seed=102),
    small_workload("gp-512", T=512, d=68, h=64, n=20, k=2, seed=103),
    small_workload("gp-513-wide", T=513, d=128, h=64, n=24, k=3, act="bf16", seed=104),
    small_workload("gp-narrow", T=2100, d=328, h=64, n=8, k=2, act="bf16", seed=105),
    small_workload("gp-quads", T=2500, d=64, h=64, n=4, k=1, seed=106),
    small_workload("gp-slices", T=3001, d=320, h=64, n=20, k=3, act="bf16", seed=107),
    small_workload("gp-72-logits", T=2200, d=136, h=64, n=36, k=2, act="bf16", seed=108),
    small_workload("gp-few-rows-wide", T=40, d=260, h=64, n=100, k=2, seed=109),
    # rows of logits and weights that are no whole quads: both, the weights only
    small_workload("gp-one-expert", T=1, d=64, h=64, n=1, k=1, seed=121),
    small_workload("gp-511-single", T=511, d=72, h=64, n=21, k=2, act="bf16", seed=122),
    small_workload("gp-512-even", T=512, d=68, h=64, n=18, k=2, seed=123),
    small_workload("gp-513-wide-single", T=513, d=128, h=64, n=23, k=3, act="bf16", seed=124),
    small_workload("gp-narrow-single", T=2100, d=328, h=64, n=7, k=2, act="bf16", seed=125),
    small_workload("gp-slices-single", T=3001, d=320, h=64, n=19, k=3, act="bf16", seed=126),
    small_workload("gp-even", T=2200, d=136, h=64, n=34, k=2, act="bf16", seed=127),
    small_workload("gp-many-single", T=2500, d=200, h=64, n=111, k=2, act="bf16", seed=128),
    small_workload("gp-few-rows-single", T=40, d=260, h=64, n=101, k=2, seed=129),
]
HIER = [
    small_workload("gp-hier", T=1500, d=128, h=64, n=64, k=4, act="bf16", a=16, k1=2, b=4, k2=2, seed=111),
    small_workload("gp-hier-odd-groups", T=700, d=64, h=64, n=60, k=4, act="bf16", a=5, k1=2, b=12, k2=2, seed=112),
    small_workload("gp-hier-few", T=100, d=64, h=64, n=160, k=2, a=8, k1=1, b=20, k2=2, seed=113),
    small_workload("gp-hier-single", T=1500, d=128, h=64, n=63, k=4, act="bf16", a=9, k1=2, b=7, k2=2, seed=114),
    small_workload("gp-hier-even", T=900, d=64, h=64, n=60, k=4, a=10, k1=2, b=6, k2=2, seed=115),
]


@pytest.mark.parametrize("w", FLAT, ids=lambda w: w.name)
def test_flat_step(w):
    check_flat(w, 0)


@pytest.mark.parametrize("w", HIER, ids=lambda w: w.name)
def test_hierarchical_step(w):
    check_hier((w,) + oracle_cached(w) + (None, None), 0)


# weight gradients of few features in many slices: 16 features, up to 32, and just above
@pytest.mark.parametrize("T,d,n,act", [(26346, 16, 20, "f32"), (20001, 8, 21, "bf16"), (40000, 8, 4, "f32"), (33000, 12, 7, "f32"), (20000, 24, 20, "bf16"), (20000, 32, 19, "f32"), (20000, 36, 20, "f32")])
def test_few_features(T, d, n, act):
    check_flat(small_workload(f"gp-features-{T}-{d}-{n}", T=T, d=d, h=64, n=n, k=2, act=act, seed=140), 0)

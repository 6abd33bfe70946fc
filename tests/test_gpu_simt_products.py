"""The float products (projection, all-float experts, gate gradients) at the borders of their tiles, slices and layouts:
whole fused steps against the oracle at the tolerances of the float paths."""
import pytest

from helpers import small_workload
from test_gpu_fused import oracle_cached, test_fused_forward_backward as check_flat
from test_gpu_hier import test_hier_fused as check_hier

pytestmark = pytest.mark.gpu

# gate widths that are no multiple of four take element-wise loads, the two gating matrices meet inside a quad; batches one
# row short of, equal to and behind a tile or a slice of the weight gradients; segments from empty to several tiles
FLAT = [
    small_workload("simt-odd-width", T=63, d=12, h=20, n=3, k=2, seed=61),
    small_workload("simt-one-tile", T=64, d=64, h=64, n=4, k=1, seed=62),
    small_workload("simt-tile-plus-one", T=65, d=68, h=132, n=5, k=2, seed=63),
    small_workload("simt-few-tokens", T=3, d=256, h=128, n=30, k=2, seed=64),
    small_workload("simt-slices", T=2049, d=36, h=40, n=6, k=2, seed=65),
    small_workload("simt-large-tiles", T=4100, d=64, h=1024, n=4, k=2, seed=66),
    small_workload("simt-bf16-rows", T=517, d=72, h=200, n=10, k=3, act="bf16", seed=67),
    small_workload("simt-bf16-gate", T=1100, d=128, h=128, n=20, k=3, act="bf16", seed=68),
]
HIER = [
    small_workload("simt-hier-odd", T=131, d=24, h=32, n=15, k=4, a=5, k1=2, b=3, k2=2, seed=71),
    small_workload("simt-hier-bf16", T=700, d=64, h=64, n=64, k=4, act="bf16", a=16, k1=2, b=4, k2=2, seed=72),
    small_workload("simt-hier-slices", T=1500, d=32, h=16, n=8, k=2, a=2, k1=1, b=4, k2=2, seed=73),
]


@pytest.mark.parametrize("w", FLAT, ids=lambda w: w.name)
def test_flat_step(w):
    check_flat(w, 0)


@pytest.mark.parametrize("w", HIER, ids=lambda w: w.name)
def test_hierarchical_step(w):
    check_hier((w,) + oracle_cached(w) + (None, None), 0)

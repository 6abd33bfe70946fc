"""bf16 expert products whose widths are multiples of eight but not of 64: last columns, contraction steps and rows of matrices behind 16, 32, 64, 128 and
256, segments of every length, and what lies behind a segment's end (infinities) must not count. Fused steps with recomputed activations."""
import pytest

from paper_1701_06538_b200 import binding as B

from helpers import small_workload
from test_gpu_fused import test_fused_forward_backward as check_flat
from test_gpu_segment_ends import test_rows_behind_a_segment_do_not_count as check_segments

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,h,scale", [(72, 200, 1), (8, 1032, 2), (136, 24, 3), (328, 264, 2), (64, 312, 1), (520, 128, 1), (248, 56, 4)])
def test_segments(d, h, scale):
    check_segments(d, h, scale, 0, 1)


@pytest.mark.parametrize("flags", [0, B.MOE_FLAG_RECOMPUTE_HID])
def test_fused_step(flags):
    check_flat(small_workload("odd-widths", T=1100, d=104, h=280, n=6, k=2, act="bf16", seed=121), flags)

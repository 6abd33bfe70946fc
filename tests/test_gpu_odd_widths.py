"""bf16 expert products whose widths are multiples of eight but not of 64: last columns, contraction steps and rows of matrices behind 16, 32, 64, 128 and
256, segments of every length, and what lies behind a segment's end (infinities) must not count. Fused steps with recomputed activations."""
import pytest
import torch

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


@pytest.mark.parametrize("rows,d,h,short", [(400000, 72, 40, 1), (511, 40, 72, 1), (512, 40, 136, 1), (513, 136, 40, 1), (1025, 264, 200, 1), (150000, 200, 264, 1),
                                            # few rows an expert on average: tiles 256 columns wide, of the long segment in two halves
                                            (40000, 264, 392, 100), (513, 520, 136, 9), (1024, 136, 120, 9)])
def test_long_weight_gradients_are_rounded_once(rows, d, h, short):
    """dW1 and dW2 of odd widths over many rows: as far from 64 bits as the rounding to bf16 alone is, within 2 %. (The operands' means are not 0: sums that grow row
    by row are what a tensor core's accumulator drops bits of; summed in one, 400000 rows were off by 1.18 times that. Sums begin anew every 512 rows.)"""
    counts = [rows] + [3] * short
    n = len(counts)
    R = sum(counts)
    cfg = B.make_config(R, d, h, n, 1, "bf16")
    g = torch.Generator(device="cuda").manual_seed(rows)
    f = lambda *s: torch.randn(*s, device="cuda", generator=g)
    offsets = torch.tensor([0] + counts, device="cuda").cumsum(0).to(torch.int32)
    xs, dys, hid = (f(R, d) + 0.5).bfloat16(), (f(R, d) + 0.5).bfloat16(), torch.relu(f(R, h)).bfloat16()
    W1, W2 = (f(n, d, h) * d ** -0.5).bfloat16(), (f(n, h, d) * h ** -0.5).bfloat16()
    ws = B.empty_bytes(B.moe_query_sizes(cfg).ws_bytes)
    out = [torch.empty_like(t) for t in (xs, W1, W1[:, 0].contiguous(), W2, W2[:, 0].contiguous())]
    B.moe_expert_ffn_bwd(cfg, xs, hid, dys, offsets, W1, W2, *out, ws)
    assert B.moe_check_status(ws) == 0
    for e, c in enumerate(counts):
        r = slice(int(offsets[e]), int(offsets[e]) + c)
        x, dy, hd = xs[r].double(), dys[r].double(), hid[r].double()
        # float sums of a few dozen or hundred products, rounded: what dz is, but for a tie or two
        dz = ((dy @ W2[e].double().t()) * (hd > 0)).bfloat16().double()
        for got, exp, ties in ((out[3][e], hd.t() @ dy, 0.0), (out[1][e], x.t() @ dz, 1e-4)):
            off = lambda t: ((t.double() - exp).square().sum() / exp.square().sum()).sqrt()
            assert off(got) <= 1.02 * off(exp.bfloat16()) + ties, (e, float(off(got)), float(off(exp.bfloat16())))

"""Products of float experts with few rows each: segments around 4, 8, 16 and 32 rows and empty ones, contractions and widths that fill no warp, every
way the products are cut, against 64 bits; infinities and NaN go where the sums of products carry them."""
import pytest
import torch

from paper_1701_06538_b200 import binding as B
from test_gpu_float_products import layer

pytestmark = pytest.mark.gpu

ENDS = [0, 1, 3, 4, 5, 7, 8, 9, 15, 16, 17, 0, 31, 32, 33, 0]


def run(counts, d, h, seed, change=lambda xs, W1: None):
    cfg, offsets, xs, dys, W1, b1, W2, b2, ws = layer(counts, d, h, seed)
    change(xs, W1)
    hid, ys = torch.full((sum(counts), h), float("nan"), device="cuda"), torch.full_like(xs, float("nan"))
    B.moe_expert_ffn(cfg, xs, offsets, W1, b1, W2, b2, hid, ys, ws)
    out = [torch.full_like(t, float("nan")) for t in (xs, W1, b1, W2, b2)]
    B.moe_expert_ffn_bwd(cfg, xs, hid, dys, offsets, W1, W2, *out, ws)
    assert B.moe_check_status(ws) == 0
    for e in range(len(counts)):
        r = slice(int(offsets[e]), int(offsets[e + 1]))
        x, dy, hd, w1, w2 = (t.double() for t in (xs[r], dys[r], hid[r], W1[e], W2[e]))
        dz = (dy @ w2.t()) * (hd > 0)
        yield e, [(hid[r], torch.relu(x @ w1 + b1[e].double())), (ys[r], hd @ w2 + b2[e].double()), (out[0][r], dz @ w1.t()),
                  (out[1][e], x.t() @ dz), (out[2][e], dz.sum(0)), (out[3][e], hd.t() @ dy), (out[4][e], dy.sum(0))]


# widths of one and three lanes, a chunk of 32 features and one more quad, narrow outputs of long contractions (the warps of a block share them), many blocks
@pytest.mark.parametrize("counts,d,h", [
    ([1], 8, 8), ([3, 0, 2], 4, 12), (ENDS, 32, 36), (ENDS, 200, 136), (ENDS, 8, 4096), (ENDS, 72, 1032), (ENDS, 1028, 60), (ENDS, 264, 392),
    (ENDS * 6, 520, 520), (ENDS * 2 + [150], 136, 264), ([2, 0, 1] * 220, 12, 20), ([5] * 9, 516, 132), ([1] * 40, 64, 2052)])
def test_against_64_bits(counts, d, h):
    for e, results in run(counts, d, h, d + h):
        for i, (got, exp) in enumerate(results):
            if exp.numel():
                err = ((got.double() - exp).abs() / (exp.abs() + exp.square().mean().sqrt() + 1e-30)).max()
                assert err <= 1e-5, (e, counts[e], i, float(err))  # the tolerance of the float layer


def test_values_that_are_no_numbers():
    def change(xs, W1):
        xs[2, 7], xs[9, 33], xs[20, 1:3] = float("inf"), float("nan"), torch.tensor([float("inf"), -float("inf")], device="cuda")
        W1[4, 5, 6] = -float("inf")

    for e, results in run(ENDS, 72, 136, 5, change):
        for i in (1, 2, 3, 5):  # (hid: the larger of NaN and 0 is 0)
            got, exp = results[i]
            assert torch.equal(got.isnan(), exp.isnan()) and torch.equal(got.isinf(), exp.isinf()), (e, i)


# a few long segments among short ones: blocks of sixteen rows and remainders in turn through both buffers; few blocks, and enough for the larger tiles
@pytest.mark.parametrize("counts,d,h", [([1403] + [2, 0, 5] * 40, 64, 64), ([0, 33, 16, 48, 1, 49, 700] + [4] * 40, 96, 136), ([17, 260, 32] + [1] * 140, 392, 520),
                                        ([65, 64, 63, 80], 72, 328), ([90] * 3 + [200], 28, 24)])
def test_uneven_loads(counts, d, h):
    for e, results in run(counts, d, h, d + h):
        for i, (got, exp) in enumerate(results):
            if exp.numel():
                err = ((got.double() - exp).abs() / (exp.abs() + exp.square().mean().sqrt() + 1e-30)).max()
                assert err <= 1e-5, (e, counts[e], i, float(err))  # the tolerance of the float layer

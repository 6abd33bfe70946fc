"""Expert products over segments of every length around the 16-row steps, 64-row blocks and 128 / 256-row tiles, on the one-CTA and
the two-CTA kernels: what lies behind a segment's last row (here infinities) must reach neither its rows nor its weight gradients."""
import pytest
import torch

from paper_1701_06538_b200 import binding as B

pytestmark = pytest.mark.gpu

ENDS = [0, 1, 15, 16, 17, 31, 33, 48, 63, 64, 65, 127, 128, 129, 191, 255, 256, 257, 300, 0]


@pytest.mark.parametrize("d,h,scale,flags,times", [(64, 128, 1, 0, 1), (192, 320, 1, 0, 1), (256, 512, 5, 0, 1),
                                                   (320, 256, 5, B.MOE_FLAG_TC_ONE_CTA, 1), (320, 256, 5, 0, 1),
                                                   # from four tiles a CTA on: weight gradients through maps of the segments
                                                   (640, 1024, 2, B.MOE_FLAG_TC_ONE_CTA, 1),
                                                   # from 32 tiles a CTA on, short segments: row products through them as well
                                                   (64, 4096, 1, 0, 8),
                                                   # the same on SM pairs
                                                   (256, 3072, 5, 0, 4)])
def test_rows_behind_a_segment_do_not_count(d, h, scale, flags, times):
    counts = []
    for c in ENDS * times:  # every segment is followed by one whose rows are infinite
        counts += [c + 256 * (scale - 1) if c else 0, 3]
    n, R = len(counts), sum(counts)
    cfg = B.make_config(R, d, h, n, 1, "bf16", flags=flags)
    S = B.moe_query_sizes(cfg)
    g = torch.Generator(device="cuda").manual_seed(d + h)
    bf = lambda *s: torch.randn(*s, device="cuda", generator=g).to(torch.bfloat16)
    offsets = torch.tensor([0] + counts, device="cuda").cumsum(0).to(torch.int32)
    xs, dys, W1, W2 = bf(R, d), bf(R, d), (bf(n, d, h) * d ** -0.5), (bf(n, h, d) * h ** -0.5)
    b1, b2 = bf(n, h), bf(n, d)
    bad = [slice(int(offsets[e]), int(offsets[e + 1])) for e in range(1, n, 2)]
    for r in bad:
        xs[r], dys[r] = float("inf"), float("inf")
    hid, ys, ws = torch.zeros_like(bf(R, h)), torch.zeros_like(xs), B.empty_bytes(S.ws_bytes)
    B.moe_expert_ffn(cfg, xs, offsets, W1, b1, W2, b2, hid, ys, ws)
    for r in bad:
        hid[r] = float("inf")
    dxs, dW1, db1, dW2, db2 = (torch.zeros_like(t) for t in (xs, W1, b1, W2, b2))
    B.moe_expert_ffn_bwd(cfg, xs, hid, dys, offsets, W1, W2, dxs, dW1, db1, dW2, db2, ws)
    assert B.moe_check_status(ws) == 0
    for e in range(0, n, 2):
        r = slice(int(offsets[e]), int(offsets[e + 1]))
        x, dy, w1, w2 = (t.double() for t in (xs[r], dys[r], W1[e], W2[e]))
        want_h = torch.relu(x @ w1 + b1[e].double())
        hd = hid[r].double()  # the stored activations are the operand
        dz = ((dy @ w2.t()) * (hd > 0)).to(torch.bfloat16).double()
        want = [(hid[r], want_h), (ys[r], hd @ w2 + b2[e].double()), (dxs[r], dz @ w1.t()), (dW1[e], x.t() @ dz), (db1[e], dz.sum(0)),
                (dW2[e], hd.t() @ dy), (db2[e], dy.sum(0))]
        for i, (got, exp) in enumerate(want):
            if exp.numel() == 0:
                continue
            rms = exp.square().mean().sqrt()
            # one rounding to bf16 (2^-9), sums of bf16-rounded terms: the bound of the other expert tests
            err = ((got.double() - exp).abs() / (exp.abs() + rms + 1e-30)).max()
            assert err <= 2e-2, (e, counts[e], i, float(err))

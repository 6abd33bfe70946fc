"""Expert products on single CTAs whose tiles are drawn at run time (from 64 a CTA on): segments of a few rows, which four records are kept ahead
for, and of more than 128. Every tile of every product has to be made once, whoever makes it."""
import pytest
import torch

from paper_1701_06538_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,h,low,high", [(5000, 64, 128, 0, 5), (1500, 64, 512, 120, 150)])
def test_every_tile_is_made(n, d, h, low, high):
    g = torch.Generator(device="cuda").manual_seed(n)
    counts = torch.randint(low, high, (n,), generator=g, device="cuda")
    counts[n // 2] = 300  # more than one row tile
    R = int(counts.sum())
    cfg = B.make_config(R, d, h, n, 1, "bf16", flags=B.MOE_FLAG_TC_ONE_CTA)
    assert (R // 128 + n) * ((h + 255) // 256) + n * (h // 128) > 64 * 148  # tiles of dz, as many as there can be, and dW2
    bf = lambda *s: torch.randn(*s, device="cuda", generator=g).to(torch.bfloat16)
    xs, dys, W1, W2, b1, b2 = bf(R, d), bf(R, d), bf(n, d, h) * d ** -0.5, bf(n, h, d) * h ** -0.5, bf(n, h), bf(n, d)
    offsets = torch.cat([counts.new_zeros(1), counts.cumsum(0)]).to(torch.int32)
    hid, ys, ws = torch.full_like(bf(R, h), float("nan")), torch.full_like(xs, float("nan")), B.empty_bytes(B.moe_query_sizes(cfg).ws_bytes)
    bits = torch.zeros(R, h // 32, dtype=torch.int32, device="cuda")
    grads = [torch.full_like(t, float("nan")) for t in (xs, W1, b1, W2, b2)]
    B.moe_expert_ffn_bits(cfg, xs, offsets, W1, b1, W2, b2, hid, ys, bits, ws)
    assert B.moe_check_status(ws) == 0
    B.moe_expert_ffn_bwd_bits(cfg, xs, hid, bits, dys, offsets, W1, W2, grads[0], grads[1], grads[2], grads[3], grads[4], ws)
    assert B.moe_check_status(ws) == 0
    e = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
    at = torch.arange(R, device="cuda") - offsets[e].long()
    width = int(counts.max())
    for lo in range(0, n, 250):  # padded to the longest segment, 250 experts at a time
        rows = (e >= lo) & (e < lo + 250)
        sl = slice(lo, min(n, lo + 250))
        pad = lambda t: torch.zeros(sl.stop - lo, width, t.shape[1], device="cuda", dtype=torch.float64).index_put((e[rows] - lo, at[rows]), t[rows].double())
        back = lambda t: t[e[rows] - lo, at[rows]]
        x, dy, hd, w1, w2 = pad(xs), pad(dys), pad(hid), W1[sl].double(), W2[sl].double()
        dz = ((dy @ w2.transpose(1, 2)) * (hd > 0)).to(torch.bfloat16).double()
        want = [(hid[rows], back(torch.relu(x @ w1 + b1[sl].double().unsqueeze(1)))), (ys[rows], back(hd @ w2 + b2[sl].double().unsqueeze(1))),
                (grads[0][rows], back(dz @ w1.transpose(1, 2))), (grads[1][sl], x.transpose(1, 2) @ dz), (grads[2][sl], dz.sum(1)),
                (grads[3][sl], hd.transpose(1, 2) @ dy), (grads[4][sl], dy.sum(1))]
        for i, (got, exp) in enumerate(want):
            # one rounding to bf16 (2^-9), sums of bf16-rounded terms: the bound of the other expert tests
            err = ((got.double() - exp).abs() / (exp.abs() + exp.square().mean().sqrt() + 1e-30)).max()
            assert err <= 2e-2, (lo, i, float(err))

"""Backward products on SM pairs take the segments by descending size: numbers of segments around those from which the order is made another way, around powers of two, and
equal sizes, against 64 bits."""
import pytest
import torch

from paper_1701_06538_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 255, 256, 257, 511, 513, 1025, 2047, 2048, 2049])
def test_segments_in_order(n):
    d = h = 64
    g = torch.Generator().manual_seed(n)
    counts = torch.randint(300, 700, (n,), generator=g)
    counts[torch.randint(0, n, (n // 3,), generator=g)] = 512  # equal ones
    if n > 100:
        counts[torch.randint(0, n, (5,), generator=g)] = 0
        counts[n // 2], counts[n - 1] = 4000, 1
    else:
        counts *= 60
    R = int(counts.sum())
    R += -R % 8  # as many tokens as eighths of the rows: a small gate
    counts[0] += R - int(counts.sum())
    assert R >= 384 * n and (R + 255) // 256 > 148  # SM pairs
    cfg = B.make_config(R // min(8, n), d, h, n, min(8, n), "bf16") if n >= 8 else B.make_config(R // 2, d, h, n, 2, "bf16")
    offsets = torch.cat([torch.zeros(1, dtype=torch.long), counts.cumsum(0)]).to(torch.int32).cuda()
    f = lambda *s, std=1.0: (torch.randn(*s, device="cuda") * std).to(torch.bfloat16)
    xs, dys, hid, W1, W2 = f(R, d), f(R, d), torch.relu(f(R, h)), f(n, d, h, std=d ** -0.5), f(n, h, d, std=h ** -0.5)
    dxs, dW1, db1, dW2, db2 = (torch.full_like(t, float("nan")) for t in (xs, W1, W1[:, 0].contiguous(), W2, W2[:, 0].contiguous()))
    ws = B.empty_bytes(B.moe_query_sizes(cfg).ws_bytes)
    B.moe_expert_ffn_bwd(cfg, xs, hid, dys, offsets, W1, W2, dxs, dW1, db1, dW2, db2, ws)
    assert B.moe_check_status(ws) == 0
    at = offsets.tolist()
    for e in list(range(0, n, max(1, n // 200))) + [n // 2, n - 1]:
        r = slice(at[e], at[e + 1])
        x, dy, hd, w1, w2 = (t.double() for t in (xs[r], dys[r], hid[r], W1[e], W2[e]))
        dz = ((dy @ w2.t()) * (hd > 0)).to(torch.bfloat16).double()
        for i, (got, exp) in enumerate(((dxs[r], dz @ w1.t()), (dW1[e], x.t() @ dz), (db1[e], dz.sum(0)), (dW2[e], hd.t() @ dy), (db2[e], dy.sum(0)))):
            if exp.numel():
                # one rounding to bf16 (2^-9), sums of bf16-rounded terms: the bound of the other expert tests
                assert ((got.double() - exp).abs() / (exp.abs() + exp.square().mean().sqrt() + 1e-30)).max() <= 2e-2, (e, i)

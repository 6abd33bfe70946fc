"""Bias gradients (sums over each expert's rows) at the expert and row counts that decide how many columns a block of their last pass
takes: few and many experts, segments of none, one and many tiles, widths that leave the last block partly empty. The
expected sums are taken in 64 bits from the tensors the call itself reads."""
import numpy as np
import pytest
import torch

from paper_1701_06538_b200 import binding as B

from helpers import host, rel_err

pytestmark = pytest.mark.gpu


def segments(n, R, skew):
    g = np.random.default_rng(n + R)
    p = 1.0 / np.arange(1, n + 1) if skew else np.ones(n)
    counts = np.floor(p / p.sum() * R).astype(np.int64)
    counts[g.integers(0, n, n // 5)] = 0
    counts[0] += R - counts.sum()
    return np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)


# tensor cores: from 128 experts on with at most 128 rows each, 1024 columns a block, else 64; others: from 1024 experts 256, else 32
@pytest.mark.parametrize("act,n,d,h,R,skew", [("bf16", 127, 64, 1088, 8000, True), ("bf16", 128, 64, 1088, 16384, True),
                                              ("bf16", 130, 128, 64, 17000, False), ("bf16", 1024, 320, 64, 30000, True),
                                              ("bf16", 1023, 72, 264, 9000, True), ("f32", 1030, 36, 300, 9000, True),
                                              ("f32", 5, 268, 44, 3000, False)])
def test_bias_gradients(act, n, d, h, R, skew):
    adt = torch.bfloat16 if act == "bf16" else torch.float32
    cfg = B.make_config(R // 2, d, h, n, 2, act)
    S, off = B.moe_query_sizes(cfg), segments(n, R, skew)
    g = torch.Generator(device="cuda").manual_seed(n)
    t = lambda *s: torch.randn(*s, device="cuda", generator=g).to(adt)
    e = lambda *s: torch.full(s, float("nan"), device="cuda", dtype=adt)
    xs, hid, dys, W1, W2 = t(R, d), t(R, h), t(R, d), t(n, d, h), t(n, h, d) * h ** -0.5
    db1, db2 = e(n, h), e(n, d)
    B.moe_expert_ffn_bwd(cfg, xs, hid, dys, torch.from_numpy(off).cuda(), W1, W2, e(R, d), e(n, d, h), db1, e(n, h, d), db2,
                         B.empty_bytes(S.ws_bytes))
    dz = np.zeros((R, h))
    y, w, m = host(dys).astype(np.float64), host(W2).astype(np.float64), host(hid) > 0
    want1, want2 = np.zeros((n, h)), np.zeros((n, d))
    for i in range(n):
        r = slice(off[i], off[i + 1])
        dz[r] = (y[r] @ w[i].T) * m[r]
        if act == "bf16":  # dz is stored rounded before it is summed
            dz[r] = torch.from_numpy(dz[r]).to(torch.bfloat16).double().numpy()
        want1[i], want2[i] = dz[r].sum(0), y[r].sum(0)
    # bf16: half an ulp of the stored sum, 2^-9, and for db1 now and then a dz that rounds the other way
    tol = 1e-2 if act == "bf16" else 1e-5
    assert rel_err(host(db2), want2)[0] <= tol and rel_err(host(db1), want1)[0] <= tol

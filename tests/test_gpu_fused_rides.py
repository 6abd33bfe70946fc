"""What rides along with other launches in the fused calls, against the stage calls that do it by itself: the same results, bit for bit, at
the sizes where riding begins or ends (chunks of 1024 slots of the dispatch index, expert counts, blocks of the last launch), and row
products of a handful of tokens in tiles half as wide."""
import numpy as np
import pytest
import torch

from helpers import TOL_BF16, assert_close, f32, host, i32
from paper_1701_06538_b200 import binding as B

pytestmark = pytest.mark.gpu


def make(T, d, h, n, k, act):
    g = torch.Generator(device="cuda")
    g.manual_seed(T + n)
    adt = torch.bfloat16 if act == "bf16" else torch.float32
    r = lambda *s, std=1.0, dtype=adt: torch.randn(*s, generator=g, device="cuda").mul_(std).to(dtype)
    fl = torch.float32
    return dict(x=r(T, d), Wg=r(d, n, std=d ** -0.5, dtype=fl), Wnoise=r(d, n, std=d ** -0.5, dtype=fl), noise=r(T, n, dtype=fl),
                W1=r(n, d, h, std=d ** -0.5), b1=r(n, h, std=0.1), W2=r(n, h, d, std=h ** -0.5), b2=r(n, d, std=0.1), dY=r(T, d)), adt


def check(T, d, h, n, k, act, backward):
    I, adt = make(T, d, h, n, k, act)
    cfg = B.make_config(T, d, h, n, k, act, 0.1, 0.1)
    S = B.moe_query_sizes(cfg)
    q = lambda *s: torch.empty(*s, device="cuda", dtype=adt)
    gate = (I["x"], I["Wg"], I["Wnoise"], I["noise"])
    weights = (I["W1"], I["b1"], I["W2"], I["b2"])
    ctx, ws = B.empty_bytes(S.ctx_bytes), B.empty_bytes(max(S.ws_bytes, S.ws_fwd_bytes, S.ws_bwd_bytes))
    ws.fill_(0xFF)
    y, losses, imp, load, counts = q(T, d), f32(2), f32(n), f32(n), i32(n)
    B.moe_forward(cfg, *gate, *weights, y, losses, imp, load, counts, ctx, ws)
    assert B.moe_check_status(ws) == 0

    idx, gates, clean, raw, kv, ki = i32(T, k), f32(T, k), f32(T, n), f32(T, n), f32(T, 2), i32(T, 2)
    xs, perm, inv, cnt, off, hid, ys, y1 = q(S.R, d), i32(S.R), i32(S.R), i32(n), i32(n + 1), q(S.R, h), q(S.R, d), q(T, d)
    losses1, imp1, load1 = f32(2), f32(n), f32(n)
    B.moe_gate(cfg, *gate, idx, gates, clean, raw, kv, ki, ws)
    B.moe_dispatch(cfg, I["x"], idx, xs, perm, inv, cnt, off, ws)
    B.moe_expert_ffn(cfg, xs, off, *weights, hid, ys, ws)
    B.moe_combine(cfg, ys, gates, inv, y1)
    B.moe_losses(cfg, idx, gates, clean, raw, kv, imp1, load1, losses1, ws)
    V = B.ctx_views(cfg, ctx)
    for a, b in ((V["topk_idx"], idx), (V["perm"], perm), (V["inv_perm"], inv), (V["offsets"], off), (counts, cnt), (V["ys"], ys), (y, y1),
                 (imp, imp1), (load, load1), (losses, losses1)):
        assert torch.equal(a, b)
    if not backward:
        return
    grads = lambda: dict(dWg=f32(d, n), dWnoise=f32(d, n), dW1=q(n, d, h), db1=q(n, h), dW2=q(n, h, d), db2=q(n, d))
    G, H, dX = grads(), grads(), q(T, d)
    ws.fill_(0xFF)
    B.moe_backward(cfg, I["dY"], *gate, *weights, ctx, dX, *G.values(), ws)
    assert B.moe_check_status(ws) == 0
    dgates, dys, dxs, dload, dXe, dXg = f32(T, k), q(S.R, d), q(S.R, d), f32(n), f32(T, d), f32(T, d)
    B.moe_combine_bwd(cfg, I["dY"], ys, gates, inv, dgates, dys)
    B.moe_expert_ffn_bwd(cfg, xs, hid, dys, off, I["W1"], I["W2"], dxs, H["dW1"], H["db1"], H["dW2"], H["db2"], ws)
    B.moe_losses_bwd(cfg, imp1, load1, idx, dgates, dload, ws)
    B.moe_gate_bwd(cfg, *gate, clean, raw, idx, gates, kv, ki, dgates, dload, H["dWg"], H["dWnoise"], dXg, ws)
    B.moe_dispatch_bwd(cfg, dxs, inv, dXe)
    for name in G:
        assert torch.equal(G[name], H[name]), name
    assert torch.equal(dX, (dXe + dXg).to(adt))


# one chunk, the last slot of a chunk, eight chunks in one launch, nine, and the largest number of experts whose index takes one pass
@pytest.mark.parametrize("R,k", [(1024, 1), (1026, 2), (8192, 4), (8196, 4)])
@pytest.mark.parametrize("n", [32, 1024, 1025])
def test_segment_plan_with_the_dispatch_index(R, k, n):
    check(R // k, 64, 64, n, k, "bf16", False)


# loss sums with the rows and the combine: up to 256 columns
@pytest.mark.parametrize("n", [31, 128, 129, 256, 257])
def test_loss_sums_with_the_row_movers(n):
    check(777, 64, 64, n, 2, "bf16", False)


# bf16, 64 x 64: 3.5 blocks an expert are left for the last launch, 1184 ride; float, 32 x 32: 2.25, the tail of a gate in slices
@pytest.mark.parametrize("n,d,h,act", [(338, 64, 64, "bf16"), (339, 64, 64, "bf16"), (526, 32, 32, "f32"), (527, 32, 32, "f32"),
                                       (8, 64, 64, "bf16"), (1024, 64, 64, "bf16")])
def test_sums_with_the_last_launch(n, d, h, act):
    check(3000, d, h, n, 2, act, True)


# products of a handful of tokens: 128 columns a tile, the last one half empty (N an odd multiple of 64), or not there at all
@pytest.mark.parametrize("d,h", [(192, 320), (320, 192), (448, 64), (64, 448)])
@pytest.mark.parametrize("T", [1, 7, 100])
def test_narrow_tiles(T, d, h):
    n, k = 6, 2
    I, adt = make(T, d, h, n, k, "bf16")
    cfg = B.make_config(T, d, h, n, k, "bf16", 0.1, 0.1)
    bounds = np.sort(np.random.default_rng(T + d).integers(0, T * k + 1, n - 1)).tolist()
    off = torch.tensor([0] + bounds + [T * k], dtype=torch.int32, device="cuda")
    xs = I["x"].repeat_interleave(k, 0).contiguous()
    hid, ys = torch.empty(T * k, h, device="cuda", dtype=adt), torch.empty(T * k, d, device="cuda", dtype=adt)
    B.moe_expert_ffn(cfg, xs, off, I["W1"], I["b1"], I["W2"], I["b2"], hid, ys, B.empty_bytes(B.moe_query_sizes(cfg).ws_bytes))
    o = off.tolist()
    for e in range(n):
        r = slice(o[e], o[e + 1])
        if o[e] == o[e + 1]:
            continue
        want = torch.relu(xs[r].double() @ I["W1"][e].double() + I["b1"][e].double())
        assert_close(host(hid[r]), want.cpu().numpy(), TOL_BF16, f"hid of {e}")
        assert_close(host(ys[r]), (hid[r].double() @ I["W2"][e].double() + I["b2"][e].double()).cpu().numpy(), TOL_BF16, f"ys of {e}")

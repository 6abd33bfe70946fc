"""hid of layers whose products go several ways: float layers (terms on the tensor cores, few rows, multiply-adds) and bf16 layers of odd widths form it as ONE chain of
multiply-adds per output in ascending order, plus the bias, rounded once. Its zeros are the ReLU mask, so that another order of the sums would now and then
move whole terms of dW1 and dX: the values are those of the oracle's chain, bit for bit, in the stage call and recomputed in a fused step."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as O
from paper_1701_06538_b200 import binding as B

pytestmark = pytest.mark.gpu


def chain(xs, W1, b1, counts):
    """[R, h] float: relu(xs . W1[e] + b1[e]) by the oracle's chain"""
    x, w, b = (np.ascontiguousarray(t.float().cpu().numpy()) for t in (xs, W1, b1))
    out, at = [], 0
    for e, c in enumerate(counts):
        if c:
            out.append(np.maximum(O.project(np.ascontiguousarray(x[at:at + c]), np.ascontiguousarray(w[e]), "f32") + b[e], np.float32(0)))
        at += c
    return torch.from_numpy(np.concatenate(out))


@pytest.mark.parametrize("counts,d,h,act", [([700, 0, 129, 64, 1], 128, 256, "f32"), ([3, 0, 17, 1], 128, 256, "f32"), ([40] * 6, 192, 64, "f32"), ([300, 200], 72, 136, "f32"),
                                            ([1500, 1400], 256, 512, "f32"), ([300, 0, 65, 1], 72, 200, "bf16"), ([20] * 7, 520, 264, "bf16"), ([1000], 136, 1032, "bf16")])
def test_stage_call(counts, d, h, act):
    n, R, dt = len(counts), sum(counts), torch.bfloat16 if act == "bf16" else torch.float32
    cfg = B.make_config(R, d, h, n, 1, act)
    g = torch.Generator(device="cuda").manual_seed(d + h + R)
    f = lambda *s, std=1.0: (torch.randn(*s, device="cuda", generator=g) * std).to(dt)
    offsets = torch.tensor([0] + counts, device="cuda").cumsum(0).to(torch.int32)
    xs, W1, b1, W2, b2 = f(R, d), f(n, d, h, std=d ** -0.5), f(n, h, std=0.1), f(n, h, d, std=h ** -0.5), f(n, d)
    hid, ys, ws = torch.empty(R, h, device="cuda", dtype=dt), torch.empty_like(xs), B.empty_bytes(B.moe_query_sizes(cfg).ws_bytes)
    B.moe_expert_ffn(cfg, xs, offsets, W1, b1, W2, b2, hid, ys, ws)
    assert B.moe_check_status(ws) == 0
    assert torch.equal(hid.cpu(), chain(xs, W1, b1, counts).to(dt))


@pytest.mark.parametrize("T,d,h,n,act", [(1500, 128, 256, 6, "f32"), (60, 128, 256, 12, "f32"), (900, 72, 200, 6, "bf16")])
def test_recomputed(T, d, h, n, act):
    """The mask of a recomputing step is that of a step that keeps hid: the same gradients, bit for bit"""
    dt, k = torch.bfloat16 if act == "bf16" else torch.float32, 2
    g = torch.Generator(device="cuda").manual_seed(T)
    f = lambda *s, std=1.0: (torch.randn(*s, device="cuda", generator=g) * std).to(dt)
    x, dY, W1, b1, W2, b2 = f(T, d), f(T, d), f(n, d, h, std=d ** -0.5), f(n, h, std=0.1), f(n, h, d, std=h ** -0.5), f(n, d, std=0.1)
    Wg, Wn, noise = (torch.randn(*s, device="cuda", generator=g) * std for s, std in (((d, n), d ** -0.5), ((d, n), d ** -0.5), ((T, n), 1.0)))
    results = []
    for flags in (0, B.MOE_FLAG_RECOMPUTE_HID):
        cfg = B.make_config(T, d, h, n, k, act, flags=flags)
        S = B.moe_query_sizes(cfg)
        ctx, ws = B.empty_bytes(S.ctx_bytes), B.empty_bytes(max(S.ws_fwd_bytes, S.ws_bwd_bytes))
        e = lambda *s, dt=torch.float32: torch.empty(*s, dtype=dt, device="cuda")
        B.moe_forward(cfg, x, Wg, Wn, noise, W1, b1, W2, b2, e(T, d, dt=dt), e(2), e(n), e(S.load_elems), e(n, dt=torch.int32), ctx, ws)
        out = [e(T, d, dt=dt), e(d, n), e(d, n)] + [torch.empty_like(t) for t in (W1, b1, W2, b2)]
        B.moe_backward(cfg, dY, x, Wg, Wn, noise, W1, b1, W2, b2, ctx, *out, ws)
        assert B.moe_check_status(ws) == 0
        results.append(out)
    for a, b in zip(*results):
        assert torch.equal(a, b)

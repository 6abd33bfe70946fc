"""The routing screen with two, four and eight lanes a row (by the number of rows) and the rows it leaves to exact chains, against the
chain everywhere: routing bit for bit, gates within what the screen's logits differ by. Groups of equal columns with equal noise
tie, so that a row has a few, up to 16 or more candidates (the whole-row route); some rows tie in all columns."""
import pytest
import torch

from paper_1701_06538_b200 import binding as B

from helpers import SCREEN_OFF, SCREEN_ON

pytestmark = pytest.mark.gpu


def routed(cfg, x, Wg, Wn, noise):
    S = B.moe_query_sizes(cfg)
    f32 = lambda m: torch.empty(m, device="cuda")
    i32 = lambda m: torch.empty(m, dtype=torch.int32, device="cuda")
    idx, gates, kv, ki = i32(S.R), f32(S.gates_elems), f32(S.kth_elems), i32(S.kth_elems)
    ws = B.empty_bytes(S.ws_bytes)
    B.moe_gate(cfg, x, Wg, Wn, noise, idx, gates, f32(S.logits_elems), f32(S.logits_elems), kv, ki, ws)
    assert B.moe_check_status(ws) == 0
    return idx, gates, ki


@pytest.mark.parametrize("T,d,n,k,hier", [(300, 64, 32, 1, None), (16383, 192, 96, 4, None), (16384, 64, 64, 3, None),
                                          (65535, 64, 32, 2, None), (65536, 128, 32, 6, None), (33000, 64, 32 * 32, 2, (32, 1, 32, 2)),
                                          (9000, 128, 32 * 96, 4, (32, 2, 96, 2)), (400, 64, 5 * 32, 2, (5, 1, 32, 2))])
def test_screened_routing_is_the_chains(T, d, n, k, hier):
    g = torch.Generator(device="cuda").manual_seed(T)
    a, k1, b, k2 = hier or (0, 0, 0, 0)
    cfgs = [B.make_config(T, d, 64, n, k, "bf16", 0.1, 0.1, a, k1, b, k2, flags=f) for f in (SCREEN_ON, SCREEN_OFF)]
    S = B.moe_query_sizes(cfgs[0])
    normal = lambda *s: torch.randn(*s, device="cuda", generator=g)
    x = normal(T, d).to(torch.bfloat16)
    x[::97] = 0.0
    Wg, Wn, noise = normal(S.wg_elems) * d ** -0.5, normal(S.wg_elems) * d ** -0.5, normal(S.logits_elems)
    width = a or n  # ties in the first gate: columns 1..4 like 0, 16..27 like 15 (where there are as many)
    for M in (Wg, Wn):
        M = M[:d * width].view(d, width)
        M[:, 1:5] = M[:, :1]
        M[:, 16:28] = M[:, 15:16]
    e = noise[:T * width].view(T, width)
    e[::2, 1:5] = e[::2, :1]
    e[1::3, 16:28] = e[1::3, 15:16]
    e[::97] = 0.0  # with the zero rows of x: every column ties
    on, off = (routed(c, x, Wg, Wn, noise) for c in cfgs)
    assert torch.equal(on[0], off[0]) and torch.equal(on[2], off[2])
    assert (on[1] - off[1]).abs().max() < 1e-5

"""The projection onto gate widths that are no multiple of four, around the 128 x 64 and 32 x 32 tiles it is cut into and the
border between the two: logits bit for bit as the oracle's chains, flat, grouped and with one matrix."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as O
from paper_1701_06538_b200 import binding as B
from paper_1701_06538_b200 import synth

from helpers import SCREEN_OFF, cat_parts, cfg_of, device_inputs, f32, host, i32, prec_of, small_workload

pytestmark = pytest.mark.gpu

# 222 tiles of 128 x 64 are the border: 14080 = 110 x 128 rows of two column tiles are short of it, 14081 are not
FLAT = [(1, 3, 1, 8, "f32"), (129, 33, 2, 40, "f32"), (14080, 33, 2, 16, "f32"), (14081, 33, 2, 20, "f32"),
        (14300, 50, 2, 24, "bf16"), (28289, 5, 1, 16, "bf16"), (9500, 65, 3, 40, "f32"), (7300, 126, 2, 8, "bf16")]


@pytest.mark.parametrize("T,n,k,d,act", FLAT)
def test_flat_logits(T, n, k, d, act):
    w = small_workload(f"width-{T}-{n}", T=T, d=d, h=16, n=n, k=k, act=act, seed=40 + k)
    check(w)


@pytest.mark.parametrize("T,a,b,act", [(300, 5, 7, "f32"), (13000, 6, 33, "f32"), (13000, 4, 35, "bf16")])
def test_grouped_logits(T, a, b, act):
    check(small_workload(f"width-{a}x{b}", T=T, d=16, h=16, n=a * b, k=2, act=act, a=a, k1=2, b=b, k2=1, seed=44))


def check(w):
    I = synth.make_all(w)
    G = O.forward(I["x"], I["Wg"], I["Wnoise"], I["noise"], I["W1"], I["b1"], I["W2"], I["b2"], w.k, w.w_importance, w.w_load,
                  prec_of(w), hier=w.hier).G
    cfg = cfg_of(w, SCREEN_OFF)
    S, D = B.moe_query_sizes(cfg), device_inputs(w, I)
    idx, gates, kv, ki = i32(w.T, w.k), f32(S.gates_elems), f32(S.kth_elems), i32(S.kth_elems)
    clean, raw = f32(S.logits_elems), f32(S.logits_elems)
    clean.fill_(float("nan")), raw.fill_(float("nan"))
    B.moe_gate(cfg, D["x"], D["Wg"], D["Wnoise"], D["noise"], idx, gates, clean, raw, kv, ki, B.empty_bytes(S.ws_bytes))
    assert (host(idx) == G.idx).all()
    levels = (G.primary, G.secondary) if w.a else (G,)
    assert (host(clean) == cat_parts([q.clean for q in levels])).all()
    assert (host(raw) == cat_parts([q.raw for q in levels])).all()


@pytest.mark.parametrize("T,n", [(14085, 15), (29000, 50)])
def test_one_matrix(T, n):
    """The balanced gate projects onto W_g alone: the same chains as those of moe_gate."""
    cfg = B.make_config(T, 24, 16, n, 1 if T % n == 0 else 2, "f32")
    S, Q = B.moe_query_sizes(cfg), B.moe_query_balanced_sizes(cfg)
    g = torch.Generator(device="cuda").manual_seed(n)
    x, Wg = torch.randn(T, 24, device="cuda", generator=g), torch.randn(24, n, device="cuda", generator=g)
    logits, clean = f32(T, n), f32(T, n)
    B.moe_gate_balanced(cfg, x, Wg, torch.full((n,), 1.0 / n, device="cuda"), logits, f32(T, n), i32(T, Q.mask_words), i32(Q.R),
                        i32(n + 1), f32(T), i32(T + 1), i32(Q.R), f32(1), i32(n), B.empty_bytes(Q.ws_bytes))
    B.moe_gate(cfg, x, Wg, Wg, torch.zeros(T, n, device="cuda"), i32(T, cfg.k), f32(T, cfg.k), clean, f32(T, n), f32(T, 2),
               i32(T, 2), B.empty_bytes(S.ws_bytes))
    assert torch.equal(logits, clean) and np.isfinite(host(logits)).all()

"""Top-k of whole rows on both sides of the row counts where its kernel stops forming the noisy logits block-wise: routing against
the oracle, bit for bit, with equal logits in many rows."""
import numpy as np
import pytest

from oracle import moe_oracle as O
from paper_1701_06538_b200 import binding as B
from paper_1701_06538_b200 import synth

from helpers import SCREEN_OFF, TOL_F32, assert_close, cfg_of, device_inputs, f32, host, i32, small_workload

pytestmark = pytest.mark.gpu


# 148 SMs x 8 rows, x n / 32 rows from 256 columns on
@pytest.mark.parametrize("n,k,border", [(33, 2, 1184), (65, 8, 1184), (130, 4, 1184), (255, 1, 1184), (288, 3, 1332), (512, 2, 2368)])
@pytest.mark.parametrize("beyond", [0, 1, 700], ids=["staged", "first-unstaged", "unstaged"])
def test_routing_around_the_border(n, k, border, beyond):
    w = small_workload(f"select-rows-{n}-{beyond}", T=border + beyond, d=8, h=16, n=n, k=k, seed=80 + k)
    I = synth.make_all(w)
    I["Wg"][:, n // 2:] = I["Wg"][:, :n - n // 2]  # equal columns: ties go to the lower index
    I["Wnoise"][:, n // 2:] = I["Wnoise"][:, :n - n // 2]
    I["noise"][::3, n // 2:] = I["noise"][::3, :n - n // 2]
    G = O.gate(I["x"], I["Wg"], I["Wnoise"], I["noise"], k, "f32")
    cfg, T = cfg_of(w, SCREEN_OFF), w.T
    S, D = B.moe_query_sizes(cfg), device_inputs(w, I)
    idx, gates, clean, raw, kv, ki = i32(T, k), f32(T, k), f32(T, n), f32(T, n), f32(T, 2), i32(T, 2)
    B.moe_gate(cfg, D["x"], D["Wg"], D["Wnoise"], D["noise"], idx, gates, clean, raw, kv, ki, B.empty_bytes(S.ws_bytes))
    assert (host(idx) == G.idx).all() and (host(ki) == G.kth_idx).all()
    assert (host(kv) == np.asarray(G.kth_val)).all()
    assert_close(host(gates), G.gates, TOL_F32, "gates")

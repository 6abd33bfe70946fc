"""Top-k of whole rows where its kernel changes its blocks (one, two, four or more warps of columns per row), with batches that
leave the last block partly empty: routing against the oracle, bit for bit."""
import numpy as np
import pytest

from oracle import moe_oracle as O
from paper_1701_06538_b200 import binding as B
from paper_1701_06538_b200 import synth

from helpers import SCREEN_OFF, TOL_F32, assert_close, cfg_of, device_inputs, f32, host, i32, small_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,n,k", [(1, 33, 1), (3, 32, 4), (5, 64, 2), (7, 65, 4), (9, 128, 8), (2, 129, 2), (257, 250, 4),
                                   (3, 1030, 3), (2, 8192, 2), (1, 40, 8)])
def test_routing_of_whole_rows(T, n, k):
    w = small_workload(f"select-{T}-{n}-{k}", T=T, d=24, h=16, n=n, k=k, seed=90 + k)
    I = synth.make_all(w)
    G = O.gate(I["x"], I["Wg"], I["Wnoise"], I["noise"], k, "f32")
    cfg = cfg_of(w, SCREEN_OFF)
    S, D = B.moe_query_sizes(cfg), device_inputs(w, I)
    idx, gates, clean, raw, kv, ki = i32(T, k), f32(T, k), f32(T, n), f32(T, n), f32(T, 2), i32(T, 2)
    B.moe_gate(cfg, D["x"], D["Wg"], D["Wnoise"], D["noise"], idx, gates, clean, raw, kv, ki, B.empty_bytes(S.ws_bytes))
    assert (host(idx) == G.idx).all() and (host(ki) == G.kth_idx).all()
    assert (host(clean) == np.asarray(G.clean)).all()
    assert_close(host(gates), G.gates, TOL_F32, "gates")

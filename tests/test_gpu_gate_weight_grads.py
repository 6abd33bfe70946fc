"""Weight gradients of the gate over row ranges, on SM pairs (d and 2n from 256 on) and on one CTA: token counts around a range's 128-row
restarts and the shortest range, widths that end inside a 256-wide tile in either direction."""
import numpy as np
import pytest

from oracle import moe_oracle as O
from paper_1701_06538_b200 import binding as B
from paper_1701_06538_b200 import synth

from helpers import TOL_F32, assert_close, cfg_of, dev, device_inputs, f32, host, oracle_run, prec_of, small_workload

pytestmark = pytest.mark.gpu

# the first two: logit gradients by 8 and by 16 lanes a row, the last block of rows not full
SHAPES = [(18949, 64, 64), (9475, 64, 96), (1, 256, 128), (127, 256, 128), (257, 320, 160), (1500, 512, 256), (6017, 576, 224), (9000, 256, 128), (3333, 192, 256), (3333, 512, 96)]


@pytest.mark.parametrize("flags", [0, B.MOE_FLAG_TC_ONE_CTA])
@pytest.mark.parametrize("T,d,n", SHAPES)
def test_gate_weight_grads(T, d, n, flags):
    w = small_workload("gate-dw", T=T, d=d, h=64, n=n, k=2, act="bf16", seed=T + d)
    I = synth.make_all(w)
    F, Bk = oracle_run(w, I)
    D, cfg, prec = device_inputs(w, I), cfg_of(w, flags), prec_of(w)
    ws = B.empty_bytes(B.moe_query_sizes(cfg).ws_bytes)
    dg, dload = O.losses_bwd(F.LS.importance, F.LS.load, F.G.idx, Bk.dgates, w.w_importance, w.w_load, prec)
    want = O.gate_bwd(I["x"], I["Wg"], I["Wnoise"], I["noise"], F.G.clean, F.G.raw, F.G.idx, F.G.gates, F.G.kth_val, F.G.kth_idx, dg, dload, prec)
    dWg, dWn, dXg = f32(d, n), f32(d, n), f32(T, d)
    B.moe_gate_bwd(cfg, D["x"], D["Wg"], D["Wnoise"], D["noise"], dev(F.G.clean), dev(F.G.raw), dev(F.G.idx), dev(F.G.gates),
                   dev(F.G.kth_val), dev(F.G.kth_idx), dev(np.asarray(dg, np.float32)), dev(np.asarray(dload, np.float32)), dWg, dWn, dXg, ws)
    assert B.moe_check_status(ws) == 0
    # the stage's own tolerance: three-term splits and sums restarted every 128 rows keep float precision
    assert_close(host(dWg), want.dWg, TOL_F32, "dWg")
    assert_close(host(dWn), want.dWnoise, TOL_F32, "dWnoise")
    assert_close(host(dXg), want.dX_gate, TOL_F32, "dX_gate")

"""The fused backward of a hierarchical layer with a slot whose row in the sorted order of the primary groups is marked as dropped in the
context: the slot is skipped, every other token's gradient is what it was."""
import pytest
import torch

from helpers import act_empty, cfg_of, device_inputs, f32, i32, small_workload
from paper_1701_06538_b200 import binding as B
from paper_1701_06538_b200 import synth

pytestmark = pytest.mark.gpu


def align(nbytes):
    return (nbytes + 255) // 256 * 256


@pytest.mark.parametrize("marker", [-1, 10 ** 9])
@pytest.mark.parametrize("k1,k2", [(1, 1), (2, 2)])
def test_a_dropped_row_of_a_secondary_gate_is_skipped(k1, k2, marker):
    w = small_workload("hier-dropped", T=600, d=64, h=64, n=1024, k=k1 * k2, a=32, k1=k1, b=32, k2=k2, act="bf16", seed=72)
    cfg = cfg_of(w)
    S, D = B.moe_query_sizes(cfg), device_inputs(w, synth.make_all(w))
    ctx, ws = B.empty_bytes(S.ctx_bytes), B.empty_bytes(max(S.ws_fwd_bytes, S.ws_bwd_bytes))
    B.moe_forward(cfg, D["x"], D["Wg"], D["Wnoise"], D["noise"], D["W1"], D["b1"], D["W2"], D["b2"], act_empty(w, w.T, w.d), f32(2),
                  f32(w.n), f32(S.load_elems), i32(w.n), ctx, ws)
    # the context ends with inv_perm_p [T * k1], counts_p [a], offsets_p [a + 1], each on 256 bytes
    at = S.ctx_bytes - align(4 * (w.a + 1)) - align(4 * w.a) - align(4 * w.T * k1)
    inv = ctx[at:at + 4 * w.T * k1].view(torch.int32)
    assert torch.equal(inv.sort().values, torch.arange(w.T * k1, device="cuda", dtype=torch.int32))

    def dX_of():
        dX = act_empty(w, w.T, w.d)
        B.moe_backward(cfg, D["dY"], D["x"], D["Wg"], D["Wnoise"], D["noise"], D["W1"], D["b1"], D["W2"], D["b2"], ctx, dX, f32(S.wg_elems),
                       f32(S.wg_elems), act_empty(w, w.n, w.d, w.h), act_empty(w, w.n, w.h), act_empty(w, w.n, w.h, w.d),
                       act_empty(w, w.n, w.d), ws)
        assert B.moe_check_status(ws) == 0
        return dX

    whole = dX_of()
    token = 77
    inv[token * k1] = marker
    dropped = dX_of()
    others = torch.arange(w.T, device="cuda") != token
    assert torch.equal(dropped[others], whole[others])
    assert torch.isfinite(dropped[token]).all() and not torch.equal(dropped[token], whole[token])

"""The workspace of a fused backward call: not much more than what the stages need one after the other beside the tensors that they hand
on. Sizes only, no GPU."""
import pytest

from paper_1701_06538_b200 import binding as B

RECOMPUTE = B.MOE_FLAG_RECOMPUTE_HID
MIB = 2 ** 20


@pytest.mark.parametrize("T,d,h,n,k,act,hier,flags", [
    (2085, 256, 512, 16, 2, "f32", None, 0),
    (3000, 128, 256, 64, 2, "f32", (8, 1, 8, 2), 0),
    (8192, 512, 1024, 32, 4, "bf16", None, 0),
    (12000, 512, 1024, 256, 4, "bf16", None, RECOMPUTE),
    (32768, 512, 1024, 256, 4, "bf16", None, 0),
    (40000, 512, 128, 1024, 2, "bf16", None, 0),
    (65536, 512, 1024, 4096, 4, "bf16", (64, 2, 64, 2), 0),
    (65536, 512, 1024, 4096, 4, "bf16", (64, 2, 64, 2), RECOMPUTE),
    (131072, 1024, 4096, 128, 2, "bf16", None, 0),
])
def test_the_fused_backward_shares_its_scratch(T, d, h, n, k, act, hier, flags):
    a, k1, b, k2 = hier or (0, 0, 0, 0)
    S = B.moe_query_sizes(B.make_config(T, d, h, n, k, act, 0.1, 0.1, a, k1, b, k2, flags))
    esz = 2 if act == "bf16" else 4
    handed_on = 2 * S.R * d * esz + 4 * (T * d + S.gates_elems)          # dys, dxs, dX of the gate, dgates
    again = S.R * h * esz if flags & RECOMPUTE else 0                    # hidden activations
    secondary = 4 * T * k1 * d if not flags & RECOMPUTE else 0           # rows of the secondary gates, kept for the last launch
    S0 = B.moe_query_sizes(B.make_config(T, d, h, n, k, act, 0.1, 0.1, a, k1, b, k2, 0))
    assert S.ws_bwd_bytes <= 1.1 * (handed_on + S0.ws_bytes + again) + secondary + 16 * MIB


@pytest.mark.parametrize("flags,most", [(0, 8192 * MIB), (RECOMPUTE, 1024 * MIB)])
@pytest.mark.parametrize("T,d,h,n,k", [(500000, 1024, 2048, 64, 2), (200000, 512, 1024, 512, 4), (40000, 1024, 4096, 32, 2), (20000, 512, 512, 32, 1), (65536, 64, 4096, 8, 4)])
def test_terms_of_float_layers_take_a_bounded_part(T, d, h, n, k, flags, most):
    """Beside what the float products need: dys, dxs, dz, recomputed hid, and the gate's gradient and scratch."""
    S = B.moe_query_sizes(B.make_config(T, d, h, n, k, "f32", 0.1, 0.1, flags=flags))
    rows = 4 * S.R * (2 * d + h + (h if flags else 0))
    gate = 4 * (T * d + 6 * S.logits_elems + S.gates_elems)
    assert S.ws_bwd_bytes <= 1.1 * (rows + gate) + most + 64 * MIB
    assert S.ws_fwd_bytes <= 1.1 * (4 * S.R * (h if flags else 0) + gate) + most + 64 * MIB

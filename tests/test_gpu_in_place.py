"""moe_expert_ffn_bwd with dxs in the place of xs: the weight gradients and dxs are those of separate buffers, bit for bit."""
import pytest
import torch

from paper_1701_06538_b200 import binding as B

pytestmark = pytest.mark.gpu


# single CTAs, with tiles dealt and (short segments) drawn; SM pairs; widths that are no multiples of 64; float layers on the tensor cores, with few rows and neither
@pytest.mark.parametrize("counts,d,h,act", [([300, 0, 17, 129] * 5, 320, 832, "bf16"), ([20] * 1500, 128, 256, "bf16"), ([900] * 40, 512, 512, "bf16"),
                                            ([300, 1, 64] * 4, 72, 520, "bf16"), ([700, 0, 300, 65], 256, 512, "f32"), ([5, 0, 17, 2], 128, 192, "f32"),
                                            ([300, 200], 72, 136, "f32")])
@pytest.mark.parametrize("odd", [False, True])
def test_dxs_in_the_place_of_xs(counts, d, h, act, odd):
    n, R, dt = len(counts), sum(counts), torch.bfloat16 if act == "bf16" else torch.float32
    cfg = B.make_config(R, d, h, n, 1, act)
    ws = B.empty_bytes(B.moe_query_sizes(cfg).ws_bytes)
    g = torch.Generator(device="cuda").manual_seed(d + h)
    f = lambda *s, std=1.0: (torch.randn(*s, device="cuda", generator=g) * std).to(dt)
    offsets = torch.tensor([0] + counts, device="cuda").cumsum(0).to(torch.int32)
    xs, dys, hid, W1, W2 = f(R, d), f(R, d), torch.relu(f(R, h)), f(n, d, h, std=d ** -0.5), f(n, h, d, std=h ** -0.5)
    if odd:  # elements that are not finite are formed from xs itself
        xs[3, 5], dys[2, 7] = float("inf"), float("nan")
    results = []
    for in_place in (False, True):
        x = xs.clone()
        out = [x if in_place else torch.full_like(xs, 7.0)] + [torch.full_like(t, 7.0) for t in (W1, W1[:, 0].contiguous(), W2, W2[:, 0].contiguous())]
        B.moe_expert_ffn_bwd(cfg, x, hid, dys, offsets, W1, W2, *out, ws)
        assert B.moe_check_status(ws) == 0
        results.append(out)
    for a, b in zip(*results):
        assert torch.equal(a.view(torch.int16 if act == "bf16" else torch.int32), b.view(torch.int16 if act == "bf16" else torch.int32))

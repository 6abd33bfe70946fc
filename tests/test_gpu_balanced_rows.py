"""Row movers of the strictly balanced layer over lists of any length (none, a few, more than a warp's 32) and widths of any number of
vectors, rows outside the range among them; the batchwise mask at the batch sizes up to which its keys stay in registers."""
import pytest
import torch

from paper_1701_06538_b200 import binding as B

from test_gpu_balanced_select import test_batchwise_mask_follows_from_the_probabilities as check_mask

pytestmark = pytest.mark.gpu

COUNTS = [0, 1, 3, 4, 5, 8, 31, 32, 33, 64, 70, 5]


@pytest.mark.parametrize("d,act", [(8, "bf16"), (256, "bf16"), (520, "bf16"), (1032, "bf16"), (4, "f32"), (264, "f32")])
def test_row_movers_over_lists(d, act):
    T, n, k = len(COUNTS), 32, 8
    R, m = T * k, T * k // n
    cfg = B.make_config(T, d, 16, n, k, act)
    adt = torch.bfloat16 if act == "bf16" else torch.float32
    tol = 2.0 ** -8 if act == "bf16" else 1e-5  # one rounding of the result; float sums of up to 70 terms
    g = torch.Generator(device="cuda").manual_seed(d)
    normal = lambda *s: torch.randn(*s, device="cuda", generator=g)
    ptr = torch.tensor([0] + COUNTS, device="cuda").cumsum(0).to(torch.int32)
    rows = torch.randint(0, R, (int(ptr[-1]),), device="cuda", generator=g, dtype=torch.int32)
    rows[::9] = -1
    rows[4::9] = R
    p, den = torch.rand(T, n, device="cuda", generator=g), 1.0 + torch.rand(T, device="cuda", generator=g)
    ys, dY, dXg = normal(R, d).to(adt), normal(T, d).to(adt), normal(T, d)
    y, dX = torch.empty(T, d, device="cuda", dtype=adt), torch.empty(T, d, device="cuda", dtype=adt)
    B.moe_combine_balanced(cfg, ys, p, den, ptr, rows, y)
    B.moe_dispatch_balanced_bwd(cfg, ys, ptr, rows, dXg, dX)
    tok = torch.randint(0, T, (R,), device="cuda", generator=g, dtype=torch.int32)
    dG, dys = torch.empty(R, device="cuda"), torch.empty(R, d, device="cuda", dtype=adt)
    B.moe_combine_balanced_bwd(cfg, dY, ys, p, den, tok, dG, dys)

    def close(got, want):
        assert (got.double() - want).abs().max() <= tol * (want.abs().max() + 1.0)

    for t in range(T):
        r = rows[int(ptr[t]):int(ptr[t + 1])].long()
        r = r[(r >= 0) & (r < R)]
        gate = (p[t, r // m] / den[t]).double().view(-1, 1)
        close(y[t], (gate * ys[r].double()).sum(0))
        close(dX[t], ys[r].double().sum(0) + dXg[t].double())
    gate = (p[tok.long(), torch.arange(R, device="cuda") // m] / den[tok.long()]).double().view(-1, 1)
    close(dys, gate * dY[tok.long()].double())
    close(dG, (dY[tok.long()].double() * ys.double()).sum(1))


# row widths on both sides of what one kernel keeps of a row (64, 128, 256), batches on both sides of 8192 and 32768 keys
@pytest.mark.parametrize("T,n,k", [(8192, 64, 2), (8255, 65, 1), (32768, 4, 1), (32769, 3, 1), (1290, 129, 4), (1028, 257, 1)])
@pytest.mark.parametrize("tied", [False, True], ids=["distinct", "tied"])
def test_batchwise_mask_at_the_borders(T, n, k, tied):
    check_mask(T, n, k, tied)

"""The batchwise mask (Eq. 18) where its kernel's sweeps end: batches around the 32 runs of a column, the batches of eight
loads, row widths on both sides of what the softmax keeps in registers; with many equal probabilities, ties to the lower
token. The expected rows follow from the probabilities the call itself returns."""
import numpy as np
import pytest
import torch

from paper_1701_06538_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,n,k", [(1, 1, 1), (8, 4, 1), (31, 31, 2), (33, 3, 2), (1024, 128, 4), (1025, 5, 5), (1056, 132, 3),
                                   (8191, 1, 1), (8256, 258, 4), (40000, 16, 2)])
@pytest.mark.parametrize("tied", [False, True], ids=["distinct", "tied"])
def test_batchwise_mask_follows_from_the_probabilities(T, n, k, tied):
    cfg = B.make_config(T, 16, 16, n, k, "f32")
    S = B.moe_query_balanced_sizes(cfg)
    g = torch.Generator(device="cuda").manual_seed(T + n)
    x = torch.randn(T, 16, device="cuda", generator=g)
    if tied:
        x = x[torch.randint(0, max(1, T // 7), (T,), device="cuda", generator=g)].contiguous()
    f32 = lambda *s: torch.full(s, -1.0, device="cuda")
    i32 = lambda *s: torch.full(s, -1, dtype=torch.int32, device="cuda")
    probs, mask, rows, thr = f32(T, n), i32(T, S.mask_words), i32(S.R), torch.full((n,), 1.0 / n, device="cuda")
    B.moe_gate_balanced(cfg, x, 0.25 * torch.randn(16, n, device="cuda", generator=g), thr, f32(T, n), probs, mask, rows,
                        i32(n + 1), f32(T), i32(T + 1), i32(S.R), f32(1), i32(n), B.empty_bytes(S.ws_bytes))
    p = probs.cpu().numpy()
    assert np.abs(p.sum(1) - 1.0).max() < 1e-5
    order = np.argsort(-p, axis=0, kind="stable")[:S.m]  # the m largest of every column, equal ones by token
    want = np.sort(order, axis=0)
    assert (rows.cpu().numpy().reshape(n, S.m) == want.T).all()
    kept = np.zeros((T, S.mask_words * 32), bool)
    kept[want.reshape(-1), np.tile(np.arange(n), S.m)] = True
    assert (np.packbits(kept, axis=1, bitorder="little").view(np.uint32) == mask.cpu().numpy().view(np.uint32)).all()

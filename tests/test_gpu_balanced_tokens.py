"""What the balanced gate sums per token and over the batch (Eq. 16, 20, the threshold counts), at the batch sizes where a warp of its
kernel takes one, two or eight tokens. The expected values follow from the probabilities and the mask the call itself
returns, in 64 bits: den and the loss differ by their rounding to float (6e-8, the loss over its absolute terms)."""
import numpy as np
import pytest
import torch

from paper_1701_06538_b200 import binding as B

from helpers import f32, host, i32

pytestmark = pytest.mark.gpu


# a warp takes T / 4736 tokens, one to eight
@pytest.mark.parametrize("T,n,k", [(7, 7, 1), (4735, 5, 2), (9471, 3, 1), (9472, 37, 1), (14208, 111, 4), (37887, 9, 3), (37888, 64, 2),
                                   (50001, 7, 1), (600, 1200, 2)])
def test_token_sums_follow_from_probabilities_and_mask(T, n, k):
    cfg = B.make_config(T, 16, 16, n, k, "f32")
    Q = B.moe_query_balanced_sizes(cfg)
    g = torch.Generator(device="cuda").manual_seed(T + n)
    x, Wg = torch.randn(T, 16, device="cuda", generator=g), 0.25 * torch.randn(16, n, device="cuda", generator=g)
    thr = (1.0 + 0.2 * torch.rand(n, device="cuda", generator=g)) / n
    probs, mask, den, loss, counts, ptr = f32(T, n), i32(T, Q.mask_words), f32(T), f32(1), i32(n), i32(T + 1)
    B.moe_gate_balanced(cfg, x, Wg, thr, f32(T, n), probs, mask, i32(Q.R), i32(n + 1), den, ptr, i32(Q.R), loss, counts,
                        B.empty_bytes(Q.ws_bytes))
    p, t = host(probs).astype(np.float64), host(thr).astype(np.float64)
    kept = np.unpackbits(mask.cpu().numpy().view(np.uint8).reshape(T, -1), axis=1, bitorder="little")[:, :n].astype(bool)
    above = host(probs) > host(thr)
    assert (host(counts) == above.sum(0)).all()
    assert (np.diff(host(ptr)) == kept.sum(1)).all() and host(ptr)[0] == 0
    want = (p * kept).sum(1)
    assert np.abs(host(den) - want).max() <= 1e-7 * max(1.0, want.max())
    terms = (above.astype(np.float64) - kept) * (p - t)
    assert abs(float(host(loss)[0]) - terms.sum()) <= 1e-7 * np.abs(terms).sum()

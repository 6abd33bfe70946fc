"""The counting sort of the dispatch on each of its routes (one chunk of 1024 slots, few histogram entries, many), at the
borders between them and with ids outside the range, against a stable sort."""
import numpy as np
import pytest
import torch

from paper_1701_06538_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,n,k", [(1, 1, 1), (31, 5, 1), (256, 8192, 4), (512, 40, 2), (1024, 33, 1), (1025, 33, 1), (5000, 1, 1),
                                   (16384, 1024, 4), (16640, 1024, 4), (3000, 1025, 4), (40000, 256, 6), (2100, 8192, 4),
                                   (1024, 1024, 1), (200, 1024, 5), (1000, 1025, 1), (8192, 1024, 1), (8193, 1024, 1), (2048, 7, 4)])
def test_dispatch_index_is_a_stable_sort(T, n, k):
    g = np.random.default_rng(T + n)
    idx = (n * g.random((T, k)) ** 3).astype(np.int32)  # skewed, repeats inside a token allowed
    bad = g.random((T, k)) < 0.01
    idx[bad] = g.choice([-1, n, 2 ** 30], size=int(bad.sum()))
    cfg = B.make_config(T, 16, 16, n, k, "bf16")
    S = B.moe_query_sizes(cfg)
    i32 = lambda m: torch.full((m,), -7, dtype=torch.int32, device="cuda")
    xs, ws = torch.empty(S.R, 16, dtype=torch.bfloat16, device="cuda"), B.empty_bytes(S.ws_bytes)
    perm, inv, counts, offsets = i32(S.R), i32(S.R), i32(n), i32(n + 1)
    B.moe_dispatch(cfg, torch.zeros(T, 16, dtype=torch.bfloat16, device="cuda"), torch.from_numpy(idx).cuda(), xs, perm, inv,
                   counts, offsets, ws)
    flat = idx.reshape(-1)
    good = np.flatnonzero((flat >= 0) & (flat < n))
    want_counts = np.bincount(flat[good], minlength=n)
    assert (counts.cpu().numpy() == want_counts).all()
    assert (offsets.cpu().numpy() == np.concatenate([[0], np.cumsum(want_counts)])).all()
    want_perm = good[np.argsort(flat[good], kind="stable")]
    assert (perm.cpu().numpy()[:good.size] == want_perm).all()
    want_inv = np.full(S.R, -1)
    want_inv[want_perm] = np.arange(good.size)
    assert (inv.cpu().numpy() == want_inv).all()

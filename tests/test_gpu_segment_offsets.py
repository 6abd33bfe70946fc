"""Expert products whose offsets end behind the batch: rows that do not exist read as zeros, whatever stands behind the tensor. The
buffers here are longer than the call is told, so that nothing outside them is touched."""
import numpy as np
import pytest
import torch

from helpers import TOL_BF16, assert_close, dev, host
from paper_1701_06538_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,n,d,h", [(600, 4, 1024, 1024),    # one CTA a tile
                                     (4096, 2, 1024, 1024),   # SM pairs
                                     (1000, 300, 64, 4096),   # one CTA a tile, segments with maps of their own
                                     (36000, 70, 256, 3072)])  # SM pairs, segments with maps of their own
def test_rows_behind_the_batch_read_as_zeros(T, n, d, h):
    over = 5
    cfg = B.make_config(T, d, h, n, 1, "bf16", 0.1, 0.1)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    bf = lambda *s: torch.randn(*s, generator=g, device="cuda").mul_(d ** -0.5).bfloat16()
    xs, W1, b1, W2, b2 = bf(T + 256, d), bf(n, d, h), bf(n, h), bf(n, h, d), bf(n, d)
    hid, ys = torch.zeros(T + 256, h, device="cuda").bfloat16(), torch.zeros(T + 256, d, device="cuda").bfloat16()
    bounds = np.linspace(0, T, n + 1).astype(np.int32)
    bounds[-1] = T + over
    B.moe_expert_ffn(cfg, xs, dev(bounds), W1, b1, W2, b2, hid, ys, B.empty_bytes(B.moe_query_sizes(cfg).ws_bytes))
    torch.cuda.synchronize()
    e = n - 1
    rows = slice(int(bounds[e]), T)
    assert_close(host(hid[rows]), host(torch.relu(xs[rows].float() @ W1[e].float() + b1[e].float())), TOL_BF16)
    # written or not, a row behind the batch holds nothing of xs
    behind = hid[T:T + over].float()
    of_zeros = torch.relu(b1[e].float()).bfloat16().float()
    assert all(torch.equal(r, of_zeros) or not r.any() for r in behind)

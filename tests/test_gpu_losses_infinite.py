"""The balancing losses of a batch with an infinite gate value: no number, like their gradient, wherever the expert stands."""
import pytest
import torch

from helpers import f32
from paper_1701_06538_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 70, 300])  # one block adds the chunks, several do, wide gates
@pytest.mark.parametrize("where", [0, 5, -1])
def test_loss_of_an_infinite_importance_is_no_number(n, where):
    T, k, e = 200, 2, where % n
    cfg = B.make_config(T, 64, 64, n, k, "f32", 0.1, 0.1)
    ws = B.empty_bytes(B.moe_query_sizes(cfg).ws_bytes)
    torch.manual_seed(1)
    clean, raw = torch.randn(T, n, device="cuda"), torch.randn(T, n, device="cuda")
    H, order = clean.topk(k + 1, dim=1)
    idx, kth = order[:, :k].int().contiguous(), H[:, k - 1:].contiguous()
    gates = H[:, :k].softmax(1).contiguous()
    idx[7, 0], idx[7, 1], gates[7, 0] = e, (e + 1) % n, float("inf")
    importance, load, losses = f32(n), f32(n), f32(2)
    B.moe_losses(cfg, idx, gates, clean, raw, kth, importance, load, losses, ws)
    assert torch.isinf(importance[e]) and torch.isfinite(importance).sum() == n - 1
    assert torch.isnan(losses[0]) and torch.isfinite(losses[1])
    dgates, dload = torch.zeros_like(gates), f32(n)
    B.moe_losses_bwd(cfg, importance, load, idx, dgates, dload, ws)
    assert torch.isnan(dgates).all() and torch.isfinite(dload).all()

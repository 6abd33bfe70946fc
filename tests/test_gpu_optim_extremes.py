"""The factored optimiser step where its running averages leave the range of ordinary floats: an expert that has had no rows for so long
that they have decayed to denormals, and an infinite gradient. Shapes of every update kernel: one launch (float and bf16), column by
column, flat."""
import numpy as np
import pytest
import torch

from helpers import cfg_of, dev, dev_act, host, small_workload
from paper_1701_06538_b200 import binding as B
from paper_1701_06538_b200 import synth

pytestmark = pytest.mark.gpu

SHAPES = [(128, 320, "bf16"), (36, 52, "f32"), (1032, 2048, "bf16"), (1088, 2056, "bf16")]


def step(w, grads, state):
    """One step from these gradients (W1, b1, W2, b2 order) and state arrays; the parameters before and after it."""
    cfg, lr, beta2, eps = cfg_of(w), 1e-2, 0.999, 1e-8
    P = [dev_act(a, w) for a in synth.make_experts(w)]
    before = [p.clone() for p in P]
    state_d = dev(np.concatenate([state[q].reshape(-1) for q in ("r1", "c1", "r2", "c2", "vb1", "vb2")]))
    B.moe_expert_adam_factored(cfg, *P, *[dev_act(g, w) for g in grads], state_d, lr, beta2, eps, 100000,
                               B.empty_bytes(B.moe_query_sizes(cfg).ws_adam_bytes))
    torch.cuda.synchronize()
    return before, P


def zeros(w):
    n, d, h = w.n, w.d, w.h
    return ([np.zeros(s, np.float32) for s in ((n, d, h), (n, h), (n, h, d), (n, d))],
            {q: np.zeros((n, s), np.float32) for q, s in (("r1", d), ("c1", h), ("r2", h), ("c2", d), ("vb1", h), ("vb2", d))})


@pytest.mark.parametrize("d,h,act", SHAPES)
@pytest.mark.parametrize("size", [1.4e-45, 1e-42, 1e-39, 1e-31, 1e-29])
def test_decayed_averages_and_no_gradient_leave_the_weights(d, h, act, size):
    w = small_workload(f"adam-decayed-{d}", T=8, d=d, h=h, n=2, k=1, act=act, seed=70)
    grads, state = zeros(w)
    for r, c in (("r1", "c1"), ("r2", "c2")):
        state[r][:] = size
        state[c][:] = size
        state[c][:, ::3] = 0.0   # units that were never active
        state[c][:, 1::3] = 1.0
    before, after = step(w, grads, state)
    for q, a, b in zip(("W1", "b1", "W2", "b2"), before, after):
        assert torch.equal(a, b), q


@pytest.mark.parametrize("d,h,act", SHAPES)
def test_an_infinite_gradient_leaves_numbers_where_the_others_are_finite(d, h, act):
    w = small_workload(f"adam-infinite-{d}", T=8, d=d, h=h, n=2, k=1, act=act, seed=71)
    grads, state = zeros(w)
    g = np.random.default_rng(5)
    for a in grads:
        a[:] = g.standard_normal(a.shape)
    grads[0][1, d // 2, h // 3] = np.inf
    grads[2][1, h // 2, d // 3] = np.inf
    _, after = step(w, grads, state)
    for q, gr, p in zip(("W1", "b1", "W2", "b2"), grads, after):
        assert np.isfinite(host(p)[np.isfinite(gr)]).all(), q

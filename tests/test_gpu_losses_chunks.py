"""The batch sums of the balancing losses at the row counts and widths that decide into how many chunks they are cut, against the
oracle."""
import numpy as np
import pytest

from oracle import moe_oracle as O
from paper_1701_06538_b200 import binding as B
from paper_1701_06538_b200 import synth

from helpers import TOL_F32, assert_close, cfg_of, dev, f32, host, small_workload

pytestmark = pytest.mark.gpu


# at most 296 chunks up to 32 columns and 16384 rows, 592 beyond
@pytest.mark.parametrize("T,n,k", [(1, 3, 1), (2368, 32, 2), (2369, 6, 2), (2369, 33, 3), (4737, 32, 4), (4737, 40, 1), (9001, 5, 5), (16384, 8, 2),
                                   (16385, 8, 2)])
def test_losses_of_whole_batches(T, n, k):
    w = small_workload(f"losses-{T}-{n}", T=T, d=16, h=16, n=n, k=k, seed=30 + k)
    I = synth.make_all(w)
    G = O.gate(I["x"], I["Wg"], I["Wnoise"], I["noise"], k, "f32")
    want = O.losses(G.idx, G.gates, G.clean, G.raw, G.kth_val, 0.1, 0.1, "f32")
    cfg = cfg_of(w)
    S = B.moe_query_sizes(cfg)
    imp, load, losses = f32(n), f32(n), f32(2)
    d = lambda a: dev(np.asarray(a, np.float32))
    B.moe_losses(cfg, dev(G.idx), d(G.gates), d(G.clean), d(G.raw), d(G.kth_val), imp, load, losses, B.empty_bytes(S.ws_bytes))
    for name, got in (("importance", imp), ("load", load), ("losses", losses)):
        assert_close(host(got), getattr(want, name), TOL_F32, name)

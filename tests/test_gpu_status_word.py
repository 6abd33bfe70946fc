"""The status word of the workspace over a whole fused call: the call's first launch clears it, and what any launch of the
call reports in it (a bounded wait that gave up) is still there when the call ends. The calls are captured into graphs; a
four-byte write of the report is put between two neighbouring launches, each pair of neighbours in turn, so that no wait has
to run out for it."""
import pytest
import torch
from cuda.bindings import driver as cu

from paper_1701_06538_b200 import binding as B
from paper_1701_06538_b200 import synth

from helpers import SCREEN_ON, act_empty, cfg_of, device_inputs, f32, i32, small_workload

pytestmark = pytest.mark.gpu

TIMEOUT = 5  # MOE_ERR_TIMEOUT
CASES = [
    (small_workload("status-f32", T=100, d=40, h=52, n=7, k=2, seed=91), 0),
    (small_workload("status-bf16", T=600, d=64, h=128, n=32, k=2, act="bf16", seed=92), SCREEN_ON),
    (small_workload("status-bf16-recompute", T=600, d=64, h=128, n=32, k=2, act="bf16", seed=92),
     SCREEN_ON | B.MOE_FLAG_RECOMPUTE_HID),
    (small_workload("status-hier", T=600, d=64, h=64, n=1024, k=2, act="bf16", a=32, k1=1, b=32, k2=2, seed=93), SCREEN_ON),
]


def check(result):
    assert result[0] == cu.CUresult.CUDA_SUCCESS, result[0]
    return result[1:]


def graph_of(fn):
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        fn()
    return g, cu.CUgraph(g.raw_cuda_graph())


def chain_of(raw):
    """the launches of a captured call in order, with the edge data between neighbours"""
    n = check(cu.cuGraphGetEdges_v2(raw, 0))[3]
    src, dst, data, n = check(cu.cuGraphGetEdges_v2(raw, n))
    after = {int(s): (d, e) for s, d, e in zip(src, dst, data)}
    assert len(after) == n, "a call on one stream is a chain"
    first = [s for s in src if int(s) not in {int(d) for d in dst}]
    assert len(first) == 1
    nodes, edges = [first[0]], []
    while int(nodes[-1]) in after:
        node, edge = after[int(nodes[-1])]
        nodes.append(node)
        edges.append(edge)
    return nodes, edges


def put_write_behind(raw, i, word):
    nodes, edges = chain_of(raw)
    check(cu.cuGraphRemoveDependencies_v2(raw, [nodes[i]], [nodes[i + 1]], [edges[i]], 1))
    p = cu.CUDA_MEMSET_NODE_PARAMS()
    p.dst, p.pitch, p.value, p.elementSize, p.width, p.height = cu.CUdeviceptr(word), 0, TIMEOUT, 4, 1, 1
    node, = check(cu.cuGraphAddMemsetNode(raw, [nodes[i]], 1, p, check(cu.cuCtxGetCurrent())[0]))
    check(cu.cuGraphAddDependencies_v2(raw, [node], [nodes[i + 1]], [cu.CUgraphEdgeData()], 1))


@pytest.mark.parametrize("w,flags", CASES, ids=[w.name for w, _ in CASES])
def test_a_report_anywhere_in_a_fused_call_survives_it(w, flags):
    cfg = cfg_of(w, flags)
    S, D = B.moe_query_sizes(cfg), device_inputs(w, synth.make_all(w))
    ctx, ws = B.empty_bytes(S.ctx_bytes), B.empty_bytes(max(S.ws_fwd_bytes, S.ws_bwd_bytes))
    args = tuple(D[q] for q in ("x", "Wg", "Wnoise", "noise", "W1", "b1", "W2", "b2"))
    keep = torch.full((w.T, w.d // 8), 0x5A, dtype=torch.uint8, device="cuda")
    out = (act_empty(w, w.T, w.d), f32(2), f32(w.n), f32(S.load_elems), i32(w.n))
    grads = (act_empty(w, w.T, w.d), f32(S.wg_elems), f32(S.wg_elems), act_empty(w, w.n, w.d, w.h), act_empty(w, w.n, w.h),
             act_empty(w, w.n, w.h, w.d), act_empty(w, w.n, w.d))
    calls = dict(forward=lambda: B.moe_forward(cfg, *args, *out, ctx, ws),
                 backward=lambda: B.moe_backward(cfg, D["dY"], *args, ctx, *grads, ws),
                 layer_forward=lambda: B.moe_layer_forward(cfg, *args, keep, 0.3, *out, ctx, ws),
                 layer_backward=lambda: B.moe_layer_backward(cfg, D["dY"], *args, keep, 0.3, ctx, *grads, ws))
    for name, call in calls.items():
        ws[:4] = TIMEOUT
        call()
        assert B.moe_check_status(ws) == 0, f"{name}: a report of an earlier call is cleared"
        g, raw = graph_of(call)
        lost, n = [], len(chain_of(raw)[0])
        for i in range(n - 1):
            g, raw = graph_of(call)
            put_write_behind(raw, i, ws.data_ptr())
            g.instantiate()
            g.replay()
            if B.moe_check_status(ws) != TIMEOUT:
                lost.append(i)
        assert not lost, f"{name}: reports behind launches {lost} of {n} are lost"

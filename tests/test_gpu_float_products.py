"""The float experts' products on the tensor cores (three bf16 terms an operand): segments around the 16-row steps, 64-row blocks and 128-row
tiles, widths of one and a half tiles, against 64 bits; infinities, NaN and sums beyond float's range come out as the chain of
fused multiply-adds gives them."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as O
from paper_1701_06538_b200 import binding as B

pytestmark = pytest.mark.gpu

ENDS = [0, 1, 15, 16, 17, 63, 64, 65, 127, 128, 129, 200, 0]


def layer(counts, d, h, seed):
    n, R = len(counts), sum(counts)
    cfg = B.make_config(R, d, h, n, 1, "f32")
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = lambda *s: torch.randn(*s, device="cuda", generator=g)
    offsets = torch.tensor([0] + counts, device="cuda").cumsum(0).to(torch.int32)
    W1, W2 = f(n, d, h) * d ** -0.5, f(n, h, d) * h ** -0.5
    return cfg, offsets, f(R, d), f(R, d), W1, f(n, h), W2, f(n, d), B.empty_bytes(B.moe_query_sizes(cfg).ws_bytes)


@pytest.mark.parametrize("d,h,pad", [(192, 320, 1300), (64, 1024, 900), (448, 64, 3000)])
def test_against_64_bits(d, h, pad):
    counts = ENDS + [pad]  # enough rows for the path (asserted: its scratch is asked for)
    cfg, offsets, xs, dys, W1, b1, W2, b2, ws = layer(counts, d, h, d + h)
    n, R = len(counts), sum(counts)
    assert B.moe_query_sizes(cfg).ws_fwd_bytes > 6 * n * d * h and B.moe_query_sizes(cfg).ws_bwd_bytes > 12 * n * d * h
    hid, ys = torch.full((R, h), float("nan"), device="cuda"), torch.full_like(xs, float("nan"))
    B.moe_expert_ffn(cfg, xs, offsets, W1, b1, W2, b2, hid, ys, ws)
    out = [torch.full_like(t, float("nan")) for t in (xs, W1, b1, W2, b2)]
    B.moe_expert_ffn_bwd(cfg, xs, hid, dys, offsets, W1, W2, *out, ws)
    assert B.moe_check_status(ws) == 0
    for e in range(n):
        r = slice(int(offsets[e]), int(offsets[e + 1]))
        x, dy, hd, w1, w2 = (t.double() for t in (xs[r], dys[r], hid[r], W1[e], W2[e]))
        dz = (dy @ w2.t()) * (hd > 0)
        want = [(hid[r], torch.relu(x @ w1 + b1[e].double())), (ys[r], hd @ w2 + b2[e].double()), (out[0][r], dz @ w1.t()),
                (out[1][e], x.t() @ dz), (out[2][e], dz.sum(0)), (out[3][e], hd.t() @ dy), (out[4][e], dy.sum(0))]
        for i, (got, exp) in enumerate(want):
            if exp.numel():
                err = ((got.double() - exp).abs() / (exp.abs() + exp.square().mean().sqrt() + 1e-30)).max()
                assert err <= 1e-5, (e, counts[e], i, float(err))  # the tolerance of the float layer


def test_values_that_are_no_numbers():
    d, h, rows = 128, 256, 1600
    cfg, offsets, xs, dys, W1, b1, W2, b2, ws = layer([rows, rows], d, h, 5)
    xs[3, 7], xs[40, 9], xs[70], xs[200, 1:3] = float("inf"), float("nan"), 3.3e38, torch.tensor([float("inf"), -float("inf")], device="cuda")
    xs[300, 0], xs[301] = 3.4e38, 1e-41  # would round beyond bf16's range; denormal
    W1[0, 5, 6] = -float("inf")
    hid, ys = torch.empty(2 * rows, h, device="cuda"), torch.empty_like(xs)
    B.moe_expert_ffn(cfg, xs, offsets, W1, b1, W2, b2, hid, ys, ws)
    assert B.moe_check_status(ws) == 0
    chain = lambda a, w: O.project(np.ascontiguousarray(a.cpu().numpy()), np.ascontiguousarray(w.cpu().numpy()), "f32")
    for got, a, w, b, relu in ((hid, xs, W1, b1, True), (ys, hid, W2, b2, False)):
        for e in range(2):
            r = slice(e * rows, e * rows + rows)
            want = chain(a[r], w[e]) + b[e].cpu().numpy()
            if relu:
                want = np.where(want > 0, want, np.float32(0))  # NaN counts as 0, as before
            have = got[r].cpu().numpy()
            finite = np.isfinite(want)
            # sums of values near float's range may or may not leave it on the way, by the order of their parts
            wide = (np.abs(a[r].cpu().numpy()) > 1e30).any(1, keepdims=True) & np.isfinite(a[r].cpu().numpy()).all(1, keepdims=True)
            assert ((np.isnan(have) == np.isnan(want)) | wide).all()
            assert ((have == want) | finite | np.isnan(want) | wide).all() and ((have == want) | np.isfinite(have) | np.isnan(have)).all()
            sound = finite & ~wide
            scale = np.abs(want) + np.sqrt(np.mean(np.square(want[sound].astype(np.float64))))
            assert (np.abs(have[sound] - want[sound]) <= 1e-5 * scale[sound]).all()


def backward(cfg, offsets, xs, hid, dys, W1, W2, ws):
    n, d, h = W1.shape
    f = lambda *s: torch.full(s, float("nan"), device="cuda")
    dxs, dW1, db1, dW2, db2 = f(*xs.shape), f(n, d, h), f(n, h), f(n, h, d), f(n, d)
    B.moe_expert_ffn_bwd(cfg, xs, hid, dys, offsets, W1, W2, dxs, dW1, db1, dW2, db2, ws)
    assert B.moe_check_status(ws) == 0
    return dxs, dW1, dW2


@pytest.mark.parametrize("counts,d,h", [([1600, 1600], 128, 256), ([130, 0, 63, 700, 1, 257], 192, 64), ([40] * 20, 64, 320)])
def test_backward_of_values_that_are_no_numbers(counts, d, h):
    cfg, offsets, xs, dys, W1, b1, W2, b2, ws = layer(counts, d, h, 9)
    n, R = len(counts), sum(counts)
    assert B.moe_query_sizes(cfg).ws_bwd_bytes > 12 * n * d * h  # the path
    inf, nan = float("inf"), float("nan")
    hid = torch.relu(torch.randn(R, h, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3)))
    row = lambda e, i: int(offsets[e]) + i
    last = n - 1
    xs[row(0, 3), 7], xs[row(0, 38), 9], xs[row(last, 2), 1:3] = inf, nan, torch.tensor([inf, -inf], device="cuda")
    dys[row(0, 5), 3], dys[row(0, 37), 60], dys[row(last, 1), 0] = nan, -inf, inf
    hid[row(0, 6), 5], hid[row(last, 4), 11] = inf, nan  # (a NaN masks: it is not above 0)
    W1[0, 5, 6], W2[last, 7, 8] = -inf, inf
    dxs, dW1, dW2 = backward(cfg, offsets, xs, hid, dys, W1, W2, ws)
    for e in range(n):
        r = slice(int(offsets[e]), int(offsets[e + 1]))
        x, dy, hd, w1, w2 = (t.double() for t in (xs[r], dys[r], hid[r], W1[e], W2[e]))
        dz = dy @ w2.t()
        dz = torch.where(hd > 0, dz, torch.zeros_like(dz))
        for i, (got, exp) in enumerate(((dxs[r], dz @ w1.t()), (dW1[e], x.t() @ dz), (dW2[e], hd.t() @ dy))):
            assert torch.equal(got.isnan(), exp.isnan()) and torch.equal(got.isposinf(), exp.isposinf()) and torch.equal(got.isneginf(), exp.isneginf()), (e, i)
            sound = exp.isfinite()
            if sound.any():
                err = (got.double() - exp).abs()[sound] / (exp.abs()[sound] + exp[sound].square().mean().sqrt() + 1e-30)
                assert err.max() <= 1e-5, (e, i, float(err.max()))  # the tolerance of the float layer


@pytest.mark.parametrize("counts,d,h", [([20000], 64, 128), ([2500] * 4, 128, 256)])
def test_a_nan_does_not_make_a_call_slow(counts, d, h):
    """Whole matrices of gradients become NaN with one value of dys. The chains that decide such elements, tile by tile, take five to six times what a
    call without takes here; element by element they took 14 and 46 times."""
    cfg, offsets, xs, dys, W1, b1, W2, b2, ws = layer(counts, d, h, 11)
    hid = torch.relu(torch.randn(sum(counts), h, device="cuda"))

    def least_ms():
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            backward(cfg, offsets, xs, hid, dys, W1, W2, ws)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    clean = least_ms()
    dys[5, 3] = float("nan")
    assert least_ms() <= 10 * clean


@pytest.mark.parametrize("of_hid,of_dys,of_w2,of_w1", [(1, 1e-36, 1, 1), (3e-37, 1, 1, 1), (1, 1e-6, 1e-30, 1), (1, 1, 1, 1e-36), (1e-30, 1e-7, 1e10, 1e-34),
                                                       (1e20, 1e14, 1e-10, 1e-8), (1, 1e30, 1, 1e-30)])
def test_operands_near_the_ends_of_floats_range(of_hid, of_dys, of_w2, of_w1):
    """Operands hold their 24 bits down to float's smallest number, and products as far up as float goes."""
    counts, d, h = [130, 0, 63, 700, 1, 257], 192, 320
    cfg, offsets, xs, dys, W1, b1, W2, b2, ws = layer(counts, d, h, 13)
    n, R = len(counts), sum(counts)
    hid = torch.relu(torch.randn(R, h, device="cuda", generator=torch.Generator(device="cuda").manual_seed(4))) * of_hid
    dys, W2, W1 = dys * of_dys, W2 * of_w2, W1 * of_w1
    for e, got in enumerate(zip(*[[t[int(offsets[e]):int(offsets[e + 1])] if i == 0 else t[e] for e in range(n)] for i, t in
                                  enumerate(backward(cfg, offsets, xs, hid, dys, W1, W2, ws))])):
        r = slice(int(offsets[e]), int(offsets[e + 1]))
        x, dy, hd, w1, w2 = (t.double() for t in (xs[r], dys[r], hid[r], W1[e], W2[e]))
        dz = (dy @ w2.t()) * (hd > 0)
        for i, exp in enumerate((dz @ w1.t(), x.t() @ dz, hd.t() @ dy)):
            rms = exp.square().mean().sqrt() if exp.numel() else 0.0
            if rms < 1e-34 * 1e-3:  # too little of float's 24 bits is left in the results themselves
                continue
            err = ((got[i].double() - exp).abs() / (exp.abs() + rms)).max()
            assert err <= 1e-5, (e, i, float(rms), float(err))  # the tolerance of the float layer


def test_a_forward_call_with_activations_near_the_least_float():
    counts, d, h = [800, 0, 700, 1, 900], 192, 320
    cfg, offsets, xs, dys, W1, b1, W2, b2, ws = layer(counts, d, h, 14)
    assert B.moe_query_sizes(cfg).ws_fwd_bytes > 6 * len(counts) * d * h  # the path
    xs, b1, b2 = xs * 1e-36, b1 * 0.0, b2 * 0.0
    hid, ys = torch.empty(sum(counts), h, device="cuda"), torch.empty_like(xs)
    B.moe_expert_ffn(cfg, xs, offsets, W1, b1, W2, b2, hid, ys, ws)
    assert B.moe_check_status(ws) == 0
    for e in (0, 2, 4):
        r = slice(int(offsets[e]), int(offsets[e + 1]))
        exp = hid[r].double() @ W2[e].double()
        assert ((ys[r].double() - exp).abs() / (exp.abs() + exp.square().mean().sqrt())).max() <= 1e-5


@pytest.mark.parametrize("d,h,scale", [(192, 320, 1), (64, 1024, 1), (448, 64, 3)])
def test_rows_behind_a_segment_do_not_count(d, h, scale):
    """Every segment is followed by one whose rows are infinite, in all operands: segments around the 16-row steps, 64-row blocks and 128-row tiles, in which the rows
    behind the end are cleared in the three terms of both operands."""
    counts = []
    for c in ENDS:
        counts += [c * scale, 3]
    counts += [900, 3]
    cfg, offsets, xs, dys, W1, b1, W2, b2, ws = layer(counts, d, h, d + h + 1)
    n, R = len(counts), sum(counts)
    hid = torch.relu(torch.randn(R, h, device="cuda", generator=torch.Generator(device="cuda").manual_seed(5)))
    assert B.moe_query_sizes(cfg).ws_bwd_bytes > 12 * n * d * h  # the path
    for e in range(1, n, 2):
        r = slice(int(offsets[e]), int(offsets[e + 1]))
        xs[r], dys[r], hid[r] = float("inf"), float("inf"), float("inf")
    dxs, dW1, dW2 = backward(cfg, offsets, xs, hid, dys, W1, W2, ws)
    for e in range(0, n, 2):
        r = slice(int(offsets[e]), int(offsets[e + 1]))
        x, dy, hd, w1, w2 = (t.double() for t in (xs[r], dys[r], hid[r], W1[e], W2[e]))
        dz = (dy @ w2.t()) * (hd > 0)
        for i, (got, exp) in enumerate(((dxs[r], dz @ w1.t()), (dW1[e], x.t() @ dz), (dW2[e], hd.t() @ dy))):
            if exp.numel():
                err = ((got.double() - exp).abs() / (exp.abs() + exp.square().mean().sqrt() + 1e-30)).max()
                assert err <= 1e-5, (e, counts[e], i, float(err))  # the tolerance of the float layer

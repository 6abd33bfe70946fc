"""The work that users of this library have it do, as cases that can be timed and compared.

Every case is one pass through the public calls of `paper_1701_06538_b200.binding`: a forward call alone, or a whole
training step (forward and backward, with the optimiser step where the model takes one). Shapes are those of the
workloads in `synth.CONFIGS`, of the paper's language models (tests/golden) and of the tests; values follow the same
distributions (x, noise, dY standard normal, weights scaled by fan-in, skewed expert loads through a constant feature),
drawn on the GPU.

kind     "forward"   moe_forward (inference: no gating noise)
         "step"      moe_forward + moe_backward
         "layer"     moe_layer_forward + moe_layer_backward (sigmoid, dropout, residual) with the hidden activations
                     recomputed, then the factored Adam step on the expert parameters
         "balanced"  a step with strictly balanced gating, composed from the stage calls
a > 0    a hierarchical layer: a groups (top k1) of b experts (top k2)
"""
import math

import torch

from paper_1701_06538_b200 import binding as B

DROP_PROB = 0.3
LR, BETA2, EPS = 1e-4, 0.999, 1e-8


def _case(name, kind, T, d, h, n, k, act="bf16", skew="none", gamma=0.0, a=0, k1=0, b=0, k2=0):
    c = dict(kind=kind, T=T, d=d, h=h, n=n, k=k, act=act, skew=skew, gamma=gamma, a=a, k1=k1, b=b, k2=k2)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a unit-test sized float layer: every kernel is a few blocks, the calls are all latency
        _case("tiny-f32-step", "step", 256, 64, 128, 8, 2, act="f32"),
        # serving: a handful of tokens through a 32-expert layer, every expert's weights read for a few rows
        _case("few-tokens-forward", "forward", 24, 512, 1024, 32, 4),
        # serving: a batch of about a thousand tokens (no round number) through a 256-expert layer
        _case("serve-batch-forward", "forward", 1019, 512, 1024, 256, 4),
        # an all-float layer of ordinary size, trained (research runs, gradient checks against other code)
        _case("f32-step", "step", 2085, 256, 512, 16, 2, act="f32"),
        # a bf16 layer whose expert count and batch are no multiples of anything
        _case("odd-sizes-step", "step", 3001, 320, 832, 20, 3),
        # the paper's language-model layer with 32 experts, training
        _case("flat-32-step", "step", 8192, 512, 1024, 32, 4),
        # the same with 256 experts in a 16 x 16 hierarchy, a small batch
        _case("hier-16x16-step", "step", 5000, 512, 1024, 256, 4, a=16, k1=2, b=16, k2=2),
        # a whole training step of the 256-expert model: layer epilogue, recomputed activations, optimiser
        _case("layer-train-256", "layer", 12000, 512, 1024, 256, 4),
        # 256 experts with loads that differ by a factor of four, training
        _case("uneven-256-step", "step", 32768, 512, 1024, 256, 4, skew="normal", gamma=0.205),
        # strictly balanced gating over the same experts, training
        _case("balanced-256-step", "balanced", 32768, 512, 1024, 256, 4, skew="normal", gamma=0.205),
        # 4096 experts in a 64 x 64 hierarchy, training: all weights read and all weight gradients written for 64 rows each
        _case("hier-64x64-step", "step", 65536, 512, 1024, 4096, 4, a=64, k1=2, b=64, k2=2),
        # a wide layer with a large batch and Zipf-distributed loads, training
        _case("wide-zipf-step", "step", 131072, 1024, 4096, 128, 2, skew="zipf", gamma=0.79),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "step", "step", "step", "step", "layer", "balanced"])
    hier = kind != "balanced" and rng.random() < 0.25
    act = "f32" if not hier and rng.random() < 0.2 else "bf16"
    unit = 8 if rng.random() < 0.15 else 64  # most layers have widths the tensor cores like, some do not
    d = unit * max(1, _log_int(rng, 64, 1024) // unit)
    h = unit * max(1, _log_int(rng, 128, 4096) // unit)
    skew, gamma = rng.choice([("none", 0.0), ("normal", 0.205), ("zipf", 0.79)])
    a = k1 = b = k2 = 0
    if hier:
        a, b = _log_int(rng, 4, 64), _log_int(rng, 4, 64)
        k1, k2 = rng.choice([(1, 2), (2, 2), (2, 3)])
        n, k = a * b, k1 * k2
    else:
        n = _log_int(rng, 4, 512)
        if rng.random() < 0.6:
            n = 32 * max(1, n // 32)
        k = min(n, rng.choice([1, 2, 2, 4, 4, 6]))
    T = _log_int(rng, 1, 20000) if kind == "forward" else _log_int(rng, 16, 60000)
    # what the matrix products, the weights and the gate of one pass may cost: well below the largest listed cases
    simt = act == "f32" or unit < 64
    plain_gate = simt or (n if not hier else a) % 32 != 0 or (hier and b % 32 != 0)
    while n * d * h > 2.5e8:
        h = max(unit, h // 2 // unit * unit)
        if h == unit:
            break
    T = min(T, int((4e10 if simt else 4e12) / (12.0 * k * d * h)))
    T = min(T, int((2e10 if plain_gate else 4e11) / (12.0 * d * ((a + k1 * b) if hier else n))), 15000 if plain_gate else T)
    T = max(T, 1)
    if kind == "balanced":  # every expert keeps k T / n examples: a whole number
        T = max(n, T // n * n)
    return _case(None, kind, T, d, h, n, k, act, skew, gamma, a, k1, b, k2)


def prepare(case, seed):
    T, d, h, n, k, a, b = (case[q] for q in ("T", "d", "h", "n", "k", "a", "b"))
    kind = case["kind"]
    train = kind != "forward"
    adt = torch.bfloat16 if case["act"] == "bf16" else torch.float32
    flags = B.MOE_FLAG_RECOMPUTE_HID if kind == "layer" else 0
    cfg = B.make_config(T, d, h, n, k, case["act"], 0.1, 0.1, a, case["k1"], b, case["k2"], flags=flags)
    S = B.moe_query_sizes(cfg)
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))

    def normal(*shape, std=1.0, dtype=torch.float32):
        t = torch.randn(*shape, generator=g, device="cuda", dtype=dtype)
        return t.mul_(std) if std != 1.0 else t

    def empty(*shape, dtype=torch.float32):
        return torch.empty(*shape, device="cuda", dtype=dtype)

    s = dict(cfg=cfg, kind=kind)
    x = normal(T, d)
    n_gate = a if a else n
    Wg = normal(S.wg_elems, std=d ** -0.5)
    if case["skew"] != "none":  # per-expert logit offsets through a constant feature
        x[:, 0] = 1.0
        if case["skew"] == "normal":
            Wg[:n_gate] = case["gamma"] * normal(n_gate)
        else:
            Wg[:n_gate] = -case["gamma"] * 1.1 * torch.log(torch.arange(1, n_gate + 1, device="cuda", dtype=torch.float32))
    s.update(x=x.to(adt), Wg=Wg, Wnoise=normal(S.wg_elems, std=d ** -0.5))
    s["noise"] = normal(S.logits_elems) if train else torch.zeros(S.logits_elems, device="cuda")
    # biases 0 as in the workloads, but those of a model in training (the optimiser divides a gradient by its own size, so
    # that a bias of 0 would become nothing but the sign of a sum that may be close to 0)
    std_b = 0.02 if kind == "layer" else 0.0
    s.update(W1=normal(n, d, h, std=d ** -0.5, dtype=adt), b1=normal(n, h, std=std_b, dtype=adt),
             W2=normal(n, h, d, std=h ** -0.5, dtype=adt), b2=normal(n, d, std=std_b, dtype=adt))
    s.update(y=empty(T, d, dtype=adt), ws=B.empty_bytes(max(S.ws_bytes, S.ws_fwd_bytes, S.ws_bwd_bytes if train else 0)))
    if kind != "balanced":
        s.update(losses=empty(2), importance=empty(n), load=empty(S.load_elems), counts=empty(n, dtype=torch.int32),
                 ctx=B.empty_bytes(S.ctx_bytes))
    if not train:
        return s
    s.update(dY=normal(T, d).to(adt), dX=empty(T, d, dtype=adt), dWg=empty(S.wg_elems), dWnoise=empty(S.wg_elems),
             dW1=empty(n, d, h, dtype=adt), db1=empty(n, h, dtype=adt), dW2=empty(n, h, d, dtype=adt), db2=empty(n, d, dtype=adt))
    if kind == "layer":
        s.update(keep=torch.randint(0, 2 ** 8, (T, d // 8), generator=g, device="cuda", dtype=torch.uint8) |
                 torch.randint(0, 2 ** 8, (T, d // 8), generator=g, device="cuda", dtype=torch.uint8),  # 3 in 4 kept
                 adam=torch.zeros(S.adam_state_elems, device="cuda"), adam_ws=B.empty_bytes(S.ws_adam_bytes), step=0)
    if kind == "balanced":
        Q = B.moe_query_balanced_sizes(cfg)
        R, i32 = Q.R, torch.int32
        s.update(thr=torch.full((n,), 1.0 / n, device="cuda"), logits=empty(T, n), probs=empty(T, n),
                 mask_bits=empty(T, Q.mask_words, dtype=i32), tok_of_row=empty(R, dtype=i32), offsets=empty(n + 1, dtype=i32),
                 den=empty(T), tok_ptr=empty(T + 1, dtype=i32), tok_rows=empty(R, dtype=i32), loss=empty(1),
                 thr_counts=empty(n, dtype=i32), gws=B.empty_bytes(Q.ws_bytes), xs=empty(R, d, dtype=adt),
                 hid=empty(R, h, dtype=adt), ys=empty(R, d, dtype=adt), dys=empty(R, d, dtype=adt), dxs=empty(R, d, dtype=adt),
                 dG_row=empty(R), dX_gate=empty(T, d), dthr=empty(n))
    return s


def _out(s, *names):
    return {q: s[q] for q in names}


def run(s):
    cfg, kind = s["cfg"], s["kind"]
    if kind == "balanced":
        B.moe_gate_balanced(cfg, s["x"], s["Wg"], s["thr"], s["logits"], s["probs"], s["mask_bits"], s["tok_of_row"], s["offsets"],
                            s["den"], s["tok_ptr"], s["tok_rows"], s["loss"], s["thr_counts"], s["gws"])
        B.moe_dispatch_balanced(cfg, s["x"], s["tok_of_row"], s["xs"])
        B.moe_expert_ffn(cfg, s["xs"], s["offsets"], s["W1"], s["b1"], s["W2"], s["b2"], s["hid"], s["ys"], s["ws"])
        B.moe_combine_balanced(cfg, s["ys"], s["probs"], s["den"], s["tok_ptr"], s["tok_rows"], s["y"])
        B.moe_combine_balanced_bwd(cfg, s["dY"], s["ys"], s["probs"], s["den"], s["tok_of_row"], s["dG_row"], s["dys"])
        B.moe_expert_ffn_bwd(cfg, s["xs"], s["hid"], s["dys"], s["offsets"], s["W1"], s["W2"], s["dxs"], s["dW1"], s["db1"],
                             s["dW2"], s["db2"], s["ws"])
        B.moe_gate_balanced_bwd(cfg, s["x"], s["Wg"], s["probs"], s["mask_bits"], s["den"], s["thr"], s["tok_ptr"], s["tok_rows"],
                                s["dG_row"], s["thr_counts"], 1.0, s["dWg"], s["dX_gate"], s["dthr"], s["gws"])
        B.moe_dispatch_balanced_bwd(cfg, s["dxs"], s["tok_ptr"], s["tok_rows"], s["dX_gate"], s["dX"])
        return _out(s, "y", "loss", "probs", "mask_bits", "tok_of_row", "thr_counts", "dX", "dWg", "dW1", "db1", "dW2", "db2", "dthr")
    weights = (s["W1"], s["b1"], s["W2"], s["b2"])
    grads = (s["dX"], s["dWg"], s["dWnoise"], s["dW1"], s["db1"], s["dW2"], s["db2"]) if kind != "forward" else ()
    results = (s["y"], s["losses"], s["importance"], s["load"], s["counts"], s["ctx"], s["ws"])
    if kind == "layer":
        B.moe_layer_forward(cfg, s["x"], s["Wg"], s["Wnoise"], s["noise"], *weights, s["keep"], DROP_PROB, *results)
        B.moe_layer_backward(cfg, s["dY"], s["x"], s["Wg"], s["Wnoise"], s["noise"], *weights, s["keep"], DROP_PROB, s["ctx"],
                             *grads, s["ws"])
        s["step"] += 1
        B.moe_expert_adam_factored(cfg, *weights, s["dW1"], s["db1"], s["dW2"], s["db2"], s["adam"], LR, BETA2, EPS, s["step"],
                                   s["adam_ws"])
        return _out(s, "y", "losses", "importance", "load", "counts", "dX", "dWg", "dWnoise", "W1", "b1", "W2", "b2", "adam")
    B.moe_forward(cfg, s["x"], s["Wg"], s["Wnoise"], s["noise"], *weights, *results)
    if kind == "forward":
        return _out(s, "y", "losses", "importance", "load", "counts")
    B.moe_backward(cfg, s["dY"], s["x"], s["Wg"], s["Wnoise"], s["noise"], *weights, s["ctx"], *grads, s["ws"])
    return _out(s, "y", "losses", "importance", "load", "counts", "dX", "dWg", "dWnoise", "dW1", "db1", "dW2", "db2")


def work(case):
    T, d, h, n, k, a, b = (case[q] for q in ("T", "d", "h", "n", "k", "a", "b"))
    kind, esz = case["kind"], 2 if case["act"] == "bf16" else 4
    R = T * k
    cols = a + case["k1"] * b if a else n               # gating columns per token
    gate_w = d * a + a * d * b if a else d * n          # elements of one gating matrix
    mats = 1 if kind == "balanced" else 2               # balanced gating has no noise matrix
    used = min(n, R)                                    # experts that get a row at all
    weights = used * (2 * d * h + d + h) * esz
    byts = T * d * esz * 2 + mats * gate_w * 4 + (T * cols * 4 if mats == 2 else 0) + weights  # x, y, gate, noise, experts
    flops = 4.0 * R * d * h + 2.0 * mats * T * d * cols
    if kind != "forward":
        byts += T * d * esz * 2 + mats * gate_w * 4 + n * (2 * d * h + d + h) * esz   # dY, dX, gate and expert gradients
        flops += 8.0 * R * d * h + 4.0 * mats * T * d * cols
    if kind == "layer":  # the keep bits; the optimiser reads and writes the parameters and its state
        byts += T * d // 8 + n * (2 * d * h + d + h) * esz + 2 * n * 3 * (d + h) * 4
    return {"bytes": float(byts), "flops": flops}


def tolerance(case):
    # Against the same layer in 64 bits (routing given), measured over the flat cases: float layers differ by 6e-7 (largest
    # 6e-6); bf16 layers by 3.2e-3, the rounding of the stored bf16 tensors. In the large bf16 layers a hidden activation
    # now and then rounds to the other side of 0 with another order of its sum, and its ReLU mask follows: single elements of
    # dW1 (largest 0.56 of the tensor's root mean square) and dX (0.17). About four times what was seen for "rel"; float sums
    # get 1e-5. Whole numbers (counts, masks, row lists) are unique and do not differ.
    if case["act"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 1e-2, "max": 0.6}


def exact(case, seed):
    """The results of `run` on these inputs in 64 bits: the layer's equations in plain torch, experts one after the other
    and differentiated by hand, the gate differentiated by autograd. Whole numbers (counts, masks, row lists) are left out:
    a routing decision between logits closer than float's resolution may fall the other way here."""
    s = prepare(case, seed)
    T, d, h, n, k, a, k1, b, k2 = (case[q] for q in ("T", "d", "h", "n", "k", "a", "k1", "b", "k2"))
    kind, f64, dev = case["kind"], torch.float64, "cuda"
    train = kind != "forward"
    x = s["x"].to(f64).requires_grad_(train)
    Wg = s["Wg"].to(f64).requires_grad_(train)
    Wn = s["Wnoise"].to(f64).requires_grad_(train and kind != "balanced")
    noise = s["noise"].to(f64)

    def cv2(v):
        return v.var(unbiased=False) / v.mean() ** 2

    def noisy_gate(x_, Wg_, Wn_, eps, kk):
        """gates and columns of the kk kept experts, P(x, i) of every column"""
        cols = Wg_.shape[1]
        clean, sigma = x_ @ Wg_, torch.nn.functional.softplus(x_ @ Wn_, threshold=700.0)
        H = clean + eps.view(-1, cols) * sigma
        top, idx = H.topk(min(kk + 1, cols), dim=1)
        if kk < cols:
            kept = torch.zeros_like(H, dtype=torch.bool).scatter_(1, idx[:, :kk], True)
            P = torch.special.ndtr((clean - torch.where(kept, top[:, kk:kk + 1], top[:, kk - 1:kk])) / sigma)
        else:
            P = torch.ones_like(H)
        return torch.softmax(top[:, :kk], dim=1), idx[:, :kk], P

    out = {}
    if kind == "balanced":  # rows: expert-major, every expert's m most probable tokens in ascending order
        m = T * k // n
        probs = torch.softmax(x @ Wg.view(d, n), dim=1)
        tok = probs.detach().topk(m, dim=0).indices.sort(dim=0).values.t().reshape(-1)
        expert = torch.arange(n, device=dev).repeat_interleave(m)
        mask = torch.zeros(T, n, device=dev, dtype=f64)
        mask[tok, expert] = 1.0
        above = (probs.detach() > s["thr"].to(f64)).to(f64)
        gate = probs[tok, expert] / (probs * mask).sum(1)[tok]
        loss = ((above - mask) * (probs - s["thr"].to(f64))).sum()
        bounds = [e * m for e in range(n + 1)]
        out.update(loss=loss.detach().view(1), probs=probs.detach(), dthr=m - above.sum(0))
    else:
        if a:
            lp, wp = T * a, d * a
            g_p, i_p, P_p = noisy_gate(x, Wg[:wp].view(d, a), Wn[:wp].view(d, a), noise[:lp], k1)
            slot_of, group = torch.arange(T * k1, device=dev), i_p.reshape(-1)
            parts, load_i = [], []
            for i in range(a):
                rows = slot_of[group == i]
                w = slice(wp + i * d * b, wp + (i + 1) * d * b)
                g, c, P = noisy_gate(x[rows // k1], Wg[w].view(d, b), Wn[w].view(d, b), noise[lp:].view(T * k1, b)[rows], k2)
                parts.append((rows, g, c + i * b))
                load_i.append(P.sum(0))
            order = torch.cat([p[0] for p in parts]).argsort()
            G = (g_p.reshape(-1, 1) * torch.cat([p[1] for p in parts])[order]).reshape(T, k)
            idx = torch.cat([p[2] for p in parts])[order].reshape(T, k)
            load_p, load_i = P_p.sum(0), torch.stack(load_i)
            sizes = torch.bincount(group, minlength=a).to(f64)
            load_h = (load_p.view(a, 1) * load_i / sizes.clamp(min=1.0).view(a, 1)).reshape(-1)
            load = torch.cat([load_h, load_p, load_i.reshape(-1), sizes])
        else:
            G, idx, P = noisy_gate(x, Wg.view(d, n), Wn.view(d, n), noise, k)
            load_h = load = P.sum(0)
        imp = torch.zeros(n, device=dev, dtype=f64).index_add(0, idx.reshape(-1), G.reshape(-1))
        losses = torch.stack([0.1 * cv2(imp), 0.1 * cv2(load_h)])
        loss = losses.sum()
        order = idx.reshape(-1).argsort(stable=True)
        tok, gate = order // k, G.reshape(-1)[order]
        bounds = [0] + torch.bincount(idx.reshape(-1), minlength=n).cumsum(0).tolist()
        out.update(losses=losses.detach(), importance=imp.detach(), load=load.detach())
    xd, g = x.detach(), gate.detach().view(-1, 1)
    W = [s[q] for q in ("W1", "b1", "W2", "b2")]

    def expert_forward(e):
        w1, b1, w2, b2 = (w[e].to(f64) for w in W)
        xe = xd[tok[bounds[e]:bounds[e + 1]]]
        he = torch.relu(xe @ w1 + b1)
        return xe, he, w1, w2, he @ w2 + b2

    ys = torch.cat([expert_forward(e)[4] for e in range(n) if bounds[e] < bounds[e + 1]])
    y = torch.zeros(T, d, device=dev, dtype=f64).index_add(0, tok, g * ys)
    out["y"] = y
    if not train:
        return {q: out.get(q) for q in ("y", "losses", "importance", "load", "counts")}
    dY = s["dY"].to(f64)
    dy = dY
    if kind == "layer":
        bits = (s["keep"].view(T, d // 8, 1) >> torch.arange(8, device=dev, dtype=torch.uint8)) & 1
        keep, sig = bits.view(T, d).to(f64) / (1.0 - DROP_PROB), torch.sigmoid(y)
        out["y"], dy = xd + keep * sig, dY * keep * sig * (1.0 - sig)
    gdt = f64 if n * d * h < 2 ** 28 else torch.float32  # 64-bit sums held in 32 bits where they would fill the card
    grads = {q: torch.zeros(s[q].shape, device=dev, dtype=gdt) for q in ("dW1", "db1", "dW2", "db2")}
    dx, dgate = torch.zeros_like(xd), (dy[tok] * ys).sum(1)
    for e in range(n):
        rows = slice(bounds[e], bounds[e + 1])
        if bounds[e] == bounds[e + 1]:
            continue
        xe, he, w1, w2, _ = expert_forward(e)
        de = g[rows] * dy[tok[rows]]
        dz = (de @ w2.t()) * (he > 0)
        grads["dW1"][e], grads["db1"][e], grads["dW2"][e], grads["db2"][e] = xe.t() @ dz, dz.sum(0), he.t() @ de, de.sum(0)
        dx.index_add_(0, tok[rows], dz @ w1.t())
    (loss + (gate * dgate).sum()).backward()
    out.update(grads, dX=dx + x.grad + (dY if kind == "layer" else 0.0), dWg=Wg.grad.view(-1))
    if kind == "balanced":
        return {q: out.get(q) for q in ("y", "loss", "probs", "mask_bits", "tok_of_row", "thr_counts", "dX", "dWg", "dW1", "db1",
                                        "dW2", "db2", "dthr")}
    out["dWnoise"] = Wn.grad.view(-1)
    if kind == "step":
        return {q: out.get(q) for q in ("y", "losses", "importance", "load", "counts", "dX", "dWg", "dWnoise", "dW1", "db1",
                                        "dW2", "db2")}
    rows, cols, full = [], [], []  # the first optimiser step: factored second moments, full ones for the biases
    for wq, bq in (("W1", "b1"), ("W2", "b2")):
        gw, gb = grads["d" + wq].to(f64), grads["d" + bq].to(f64)
        r, c, v = ((1.0 - BETA2) * (gw ** 2).mean(2), (1.0 - BETA2) * (gw ** 2).mean(1), (1.0 - BETA2) * gb ** 2)
        vh = r.unsqueeze(2) * c.unsqueeze(1) / r.mean(1).clamp(min=1e-300).view(n, 1, 1) / (1.0 - BETA2)
        out[wq] = s[wq].to(f64) - LR * gw / (vh.sqrt() + EPS)
        out[bq] = s[bq].to(f64) - LR * gb / ((v / (1.0 - BETA2)).sqrt() + EPS)
        rows.append(r), cols.append(c), full.append(v)
    out["adam"] = torch.cat([q.reshape(-1) for q in (rows[0], cols[0], rows[1], cols[1], full[0], full[1])])
    return {q: out.get(q) for q in ("y", "losses", "importance", "load", "counts", "dX", "dWg", "dWnoise", "W1", "b1", "W2", "b2",
                                    "adam")}

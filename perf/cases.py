"""Timed cases of the FastMMoE MoE layer: what a serving program asks of this library, through its Python binding.

Layer shapes are those of the workloads in `paper_2511_17885_b200.inputs`: a Qwen3-MoE-style layer (128 experts,
top-8, 4 for vision tokens), a DeepSeekMoE-style layer (64 experts, top-6, 3 for vision tokens, two shared experts, a
skewed load through the router bias) and the small fp32 layer of the correctness workload.  A sequence is `n_vis`
vision tokens, 16 x 16 patches a tile in raster order (the last tile may be cut short), followed by `n_text` text
tokens; `shrink` takes that many vision tokens off each further sequence of the batch.

kinds:
  layer        one MoE layer (fmmoe_moe_forward)
  layer_prune  the layer and one pruning stage on its output (fmmoe_moe_forward_prune)
  stage        a pruning stage guided by attention: fmmoe_attention_importance, then fmmoe_prune_visual
  stack        several residual layers, vision tokens on K_v experts from the second on (fmmoe_stack_forward)
"""
import math

import torch

from paper_2511_17885_b200 import binding as B

_SHAPES = {
    "qwen": dict(dtype="bf16", hidden=2048, experts=128, inter=768, n_shared=0, top_k=8, top_k_vis=4, bias_std=0.0),
    "deepseek": dict(dtype="bf16", hidden=2048, experts=64, inter=1408, n_shared=2, top_k=6, top_k_vis=3, bias_std=0.5),
    "tiny": dict(dtype="f32", hidden=256, experts=8, inter=512, n_shared=0, top_k=2, top_k_vis=1, bias_std=0.0),
}
_NO_PRUNE = dict(window=0, gamma=0.0, alpha=1.0, retain=1.0, attn=False)
_HEADS, _KV_HEADS, _HEAD_DIM = 16, 4, 64


def _case(kind, shape, n_vis, n_text, batch=1, shrink=0, fp8=False, residual=False, n_layers=1, **prune):
    c = dict(kind=kind, shape=shape, n_vis=n_vis, n_text=n_text, batch=batch, shrink=shrink, fp8=fp8,
             residual=residual, n_layers=n_layers)
    c.update(_NO_PRUNE)
    c.update(prune)
    return c


def listed():
    named = {
        # one sequence decoding its next token: six routed and two shared experts are read for a single row
        "decode 1": _case("layer", "deepseek", 0, 1, residual=True),
        # a decode step of a batch of 16 sequences: most experts get a row or two
        "decode 16": _case("layer", "qwen", 0, 16, residual=True),
        # a short prefill chunk, one thumbnail image cut to 136 patches and a prompt
        "chunk 200": _case("layer", "deepseek", 136, 64, residual=True),
        # an odd-sized prompt: two whole tiles, a cut one, and text; merged and dropped windows by attention
        "ragged 686": _case("layer_prune", "qwen", 611, 75, window=5, gamma=0.05, alpha=0.6, retain=0.5, attn=True),
        # prefill of one multimodal prompt, either backbone family, followed by its pruning stage
        "prefill deepseek": _case("layer_prune", "deepseek", 2304, 128, window=3, gamma=0.05, alpha=0.9, retain=0.5),
        "prefill qwen": _case("layer_prune", "qwen", 3328, 256, window=5, gamma=0.025, alpha=0.5, retain=0.75, attn=True),
        # the same prompt with the expert matrices stored in FP8
        "prefill qwen fp8": _case("layer_prune", "qwen", 3328, 256, fp8=True, window=5, gamma=0.05, alpha=0.6, retain=0.5),
        # batched prefill: the benchmark's batch of four, and a batch of eight in the middle of a residual stack
        "batch 4 qwen": _case("layer_prune", "qwen", 3328, 256, batch=4, window=5, gamma=0.05, alpha=0.6, retain=0.5),
        "batch 8 deepseek": _case("layer", "deepseek", 2304, 128, batch=8, residual=True),
        # fp32 layer (correctness workload), pruned
        "fp32 256": _case("layer_prune", "tiny", 224, 32, window=5, gamma=0.05, alpha=0.6, retain=0.5),
        # attention-guided pruning of a batch whose layer ran elsewhere, sequences of different lengths
        "stage batch 8": _case("stage", "deepseek", 2304, 128, batch=8, shrink=17, window=3, gamma=0.2, alpha=0.7,
                               retain=0.25, attn=True),
        # a whole call over several layers, expert reduction only
        "stack 4": _case("stack", "qwen", 3328, 256, n_layers=4),
    }
    return [dict(c, name=n) for n, c in named.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: 1 to 16,384 tokens in a call (log-uniform), either family, every kind but the stack."""
    window = rng.choice((3, 5))
    prune = dict(window=window, gamma=rng.choice((0.025, 0.05, 0.1, 0.2)), alpha=round(rng.uniform(0.3, 1.0), 2),
                 retain=round(rng.uniform(0.25, 0.75), 3), attn=rng.random() < 0.5)
    pick = rng.random()
    if pick < 0.12:
        n = _log_int(rng, 24, 1024)
        n_text = max(1, int(n * rng.uniform(0.05, 0.3)))
        return _case("layer_prune", "tiny", n - n_text, n_text, **prune)
    shape = rng.choice(("qwen", "deepseek"))
    if pick < 0.24:
        batch = rng.randint(1, 8)
        n = _log_int(rng, 256, 3000)
        n_text = max(1, int(n * rng.uniform(0.03, 0.2)))
        return _case("stage", shape, n - n_text, n_text, batch=batch, shrink=rng.randint(0, n // 32), **dict(prune, attn=True))
    if pick < 0.44:      # decode steps: text rows only
        return _case("layer", shape, 0, _log_int(rng, 1, 255), fp8=rng.random() < 0.25, residual=True)
    batch = rng.randint(1, 4)
    n = max(24, _log_int(rng, 64, 16384) // batch)
    n_text = max(1, int(n * rng.uniform(0.03, 0.3)))
    fp8 = rng.random() < 0.2
    shrink = rng.randint(0, n // 32)
    if pick < 0.62:
        return _case("layer", shape, n - n_text, n_text, batch=batch, shrink=shrink, fp8=fp8, residual=True)
    return _case("layer_prune", shape, n - n_text, n_text, batch=batch, shrink=shrink, fp8=fp8, **prune)


# ---------------------------------------------------------------------------------------------- inputs
def _layout(case):
    """Vision tokens of each sequence, and the token offsets."""
    n_vis = [max(0, case["n_vis"] - b * case["shrink"]) for b in range(case["batch"])]
    off = [0]
    for v in n_vis:
        off.append(off[-1] + v + case["n_text"])
    return n_vis, off


def _retain(case, n_vis):
    return [int(math.floor(v * case["retain"] + 1e-9)) for v in n_vis]


def _smoother(device, n=16, sigma=2.0):
    """[n, n] matrix of a Gaussian filter over n patches with a mirrored border."""
    r = int(4 * sigma)
    k = torch.exp(-0.5 * (torch.arange(-r, r + 1, dtype=torch.float64) / sigma) ** 2)
    k /= k.sum()
    m = torch.zeros(n, n, dtype=torch.float64)
    for i in range(n):
        for d in range(-r, r + 1):
            j = (i + d) % (2 * n)
            m[i, j if j < n else 2 * n - 1 - j] += k[d + r]
    return m.to(device=device, dtype=torch.float32)


def _patches(g, n_vis, channels, noise):
    """[n_vis, channels]: neighbouring patches of a tile are alike (unit variance per tile and channel, plus noise)."""
    n_tiles = -(-n_vis // 256)
    m = _smoother("cuda")
    f = torch.randn(n_tiles, 16, 16, channels, device="cuda", generator=g)
    f = torch.einsum("ij,tjkc,lk->tilc", m, f, m)
    f = f - f.mean(dim=(1, 2), keepdim=True)
    f = f / (f.std(dim=(1, 2), keepdim=True, unbiased=False) + 1e-12)
    f = f + noise * torch.randn(f.shape, device="cuda", generator=g)
    return f.reshape(n_tiles * 256, channels)[:n_vis]


def _tokens(g, case, hidden, dtype):
    n_vis, off = _layout(case)
    rows, mask = [], torch.zeros(off[-1], dtype=torch.uint8, device="cuda")
    for b, v in enumerate(n_vis):
        if v:
            rows.append(_patches(g, v, hidden, 0.1).to(dtype))
            mask[off[b]:off[b] + v] = 1
        rows.append(torch.randn(case["n_text"], hidden, device="cuda", generator=g).to(dtype))
    return torch.cat(rows).contiguous(), mask


def _to_fp8(w):
    """[G, R, C] -> FP8 E4M3 bytes and the exponents of the power-of-two scales of their 128 x 128 blocks."""
    G, R, C = w.shape
    blocks = w.float().view(G, R // 128, 128, C // 128, 128)
    e = torch.ceil(torch.log2(blocks.abs().amax(dim=(2, 4)) / 448.0)).clamp_(-100, 7)
    q = (blocks / torch.exp2(e)[:, :, None, :, None]).to(torch.float8_e4m3fn)
    return q.view(torch.uint8).reshape(G, R, C).contiguous(), e.to(torch.int8).contiguous()


def _weights(g, case, down_std=0.02):
    s = _SHAPES[case["shape"]]
    dt = torch.bfloat16 if s["dtype"] == "bf16" else torch.float32
    H, E, I, Ns = s["hidden"], s["experts"], s["inter"], s["n_shared"]

    def normal(*shape, std=0.02):
        return torch.empty(shape, dtype=dt, device="cuda").normal_(0.0, std, generator=g)

    w = {"router_w": normal(E, H), "router_b": None, "w_gate": normal(E, I, H), "w_up": normal(E, I, H),
         "w_down": normal(E, H, I, std=down_std)}
    if s["bias_std"]:
        w["router_b"] = torch.empty(E, device="cuda").normal_(0.0, s["bias_std"], generator=g)
    if Ns:
        w.update(ws_gate=normal(Ns, I, H), ws_up=normal(Ns, I, H), ws_down=normal(Ns, H, I, std=down_std))
    if case["fp8"]:
        for k in [k for k in w if k.startswith(("w_", "ws_"))]:
            w[k], w[k + "_scale"] = _to_fp8(w[k])
    return w


_handle = None


def _the_handle():
    global _handle
    if _handle is None:
        _handle = B.Handle(0)       # one handle for the program's life, as its caller keeps
    return _handle


def _inputs(case, seed):
    """Everything the call reads, as tensors; the same for the same seed."""
    s = _SHAPES[case["shape"]]
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 11)
    dt = torch.bfloat16 if s["dtype"] == "bf16" else torch.float32
    d = {}
    d["x"], d["mask"] = _tokens(g, case, s["hidden"], dt)
    n_vis, off = _layout(case)
    if case["kind"] == "stage":
        # routing probabilities and output rows of a layer that has run, its last queries and its keys
        logits = d["x"].float() @ torch.empty(s["hidden"], s["experts"], device="cuda").normal_(0.0, 0.02, generator=g)
        d["probs"] = torch.softmax(logits, dim=1)
        d["q"] = torch.randn(case["batch"], _HEADS, _HEAD_DIM, device="cuda", generator=g).to(dt)
        walk = torch.cumsum(0.15 * torch.randn(off[-1], _KV_HEADS, _HEAD_DIM, device="cuda", generator=g), dim=0)
        d["k"] = (walk / (walk.abs().max() + 1e-9) * 3.0
                  + 0.3 * torch.randn(walk.shape, device="cuda", generator=g)).to(dt)
        return d
    # down-projections of a residual stack carry the usual 1 / sqrt(2 layers), else its activations grow without bound
    down = 0.02 / math.sqrt(2.0 * 24) if case["kind"] == "stack" else 0.02
    d["w"] = [_weights(g, case, down) for _ in range(case["n_layers"])]
    d["attn"] = None
    if case["attn"]:
        d["attn"] = torch.zeros(off[-1], device="cuda")
        for b, v in enumerate(n_vis):
            if v:
                d["attn"][off[b]:off[b] + v] = torch.softmax(_patches(g, v, 1, 0.3)[:, 0], dim=0)
    return d


def prepare(case, seed):
    s = _SHAPES[case["shape"]]
    d = _inputs(case, seed)
    n_vis, off = _layout(case)
    st = {"case": case, "h": _the_handle(), "in": d, "n_vis": n_vis, "off": off, "n_retain": _retain(case, n_vis)}
    if case["window"]:
        st["pp"] = B.prune_params(case["window"], case["gamma"], case["alpha"])
    if case["kind"] == "stage":
        return st
    st["flags"] = B.FLAG_REDUCE_ON | (B.FLAG_RESIDUAL if case["residual"] else 0)
    st["desc"] = B.make_desc(s["hidden"], s["experts"], s["inter"], s["n_shared"], s["inter"] if s["n_shared"] else 0,
                             s["top_k"], s["top_k_vis"], d["x"].dtype,
                             B.WEIGHTS_FP8_BLOCK128 if case["fp8"] else B.WEIGHTS_AS_DTYPE)
    st["w"] = [B.make_weights(w) for w in d["w"]]
    T = off[-1]
    st["out"] = torch.empty_like(d["x"])
    st["route"] = {"probs": torch.empty(T, s["experts"], device="cuda"),
                   "topk_idx": torch.empty(T, s["top_k"], dtype=torch.int32, device="cuda")}
    return st


def run(st):
    c, h, d = st["case"], st["h"], st["in"]
    if c["kind"] == "stage":
        attn = h.fmmoe_attention_importance(d["q"], d["k"], st["off"])
        r = h.fmmoe_prune_visual(st["pp"], d["probs"], attn, d["x"], d["mask"], st["off"], st["n_vis"], st["n_retain"])
        return {"attn": attn, "x_out": r["x_out"], "keep_idx": r["keep_idx"], "kind": r["kind"],
                "is_visual_out": r["is_visual_out"]}
    if c["kind"] == "stack":
        x_out, mask, _ = h.fmmoe_stack_forward(st["desc"], st["w"], 1, [], d["x"], d["mask"], st["off"], st["n_vis"])
        return {"x_out": x_out, "is_visual_out": mask}
    if c["kind"] == "layer":
        return {"out": h.fmmoe_moe_forward(st["desc"], st["w"][0], d["x"], d["mask"], st["flags"], out=st["out"])}
    r = h.fmmoe_moe_forward_prune(st["desc"], st["w"][0], d["x"], d["mask"], st["flags"], st["out"], st["route"], st["pp"],
                                  d["attn"], st["off"], st["n_vis"], st["n_retain"])
    return {"out": st["out"], "probs": st["route"]["probs"], "topk_idx": st["route"]["topk_idx"], "x_out": r["x_out"],
            "keep_idx": r["keep_idx"], "kind": r["kind"], "is_visual_out": r["is_visual_out"]}


# ---------------------------------------------------------------------------------------------- what it has to do
def _kept(case, v, eta):
    """(tokens kept, merged windows) of a sequence with v vision tokens pruned towards eta."""
    W = case["window"]
    if not W or v - eta <= W:
        return v, 0
    m = min(int(math.floor(eta * case["gamma"] + 1e-9)), (v - eta) // (W - 1), v // W)
    d = min((v - eta - m * (W - 1)) // W, v // W - m)
    return v - m * (W - 1) - d * W, m


def work(case):
    s = _SHAPES[case["shape"]]
    H, E, I, Ns, K, Kv = s["hidden"], s["experts"], s["inter"], s["n_shared"], s["top_k"], s["top_k_vis"]
    n_vis, off = _layout(case)
    T, V, e = off[-1], sum(n_vis), 2 if s["dtype"] == "bf16" else 4
    kept, merged = zip(*(_kept(case, v, r) for v, r in zip(n_vis, _retain(case, n_vis))))
    T_out = T - V + sum(kept)
    prune_bytes = (T_out + sum(merged) * (max(case["window"], 1) - 1)) * H * e + T_out * (H * e + 6) + V * E * 4
    if case["kind"] == "stage":
        kv = T * _KV_HEADS * _HEAD_DIM * e
        return {"bytes": prune_bytes + kv + T * 5, "flops": 2 * T * _HEADS * _HEAD_DIM}
    bytes_, flops = 0, 0
    for layer in range(case["n_layers"]):
        kv = Kv if case["kind"] != "stack" or layer >= 1 else K
        pairs = V * kv + (T - V) * K
        # experts that any token picks: text tokens choose for themselves, a tile of vision tokens much alike
        touched = E * (1.0 - (1.0 - K / E) ** (T - V) * (1.0 - kv / E) ** (V / 16))
        we = 1 if case["fp8"] else e
        bytes_ += (touched + Ns) * 3 * H * I * we + E * H * e + 2 * T * H * e + T
        flops += 6 * H * I * (pairs + Ns * T) + 2 * T * H * E
    if case["kind"] == "layer_prune":
        bytes_ += prune_bytes + T * E * 4 + T * K * 4
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """About four times the error against `exact` that the library shows (2.9e-3 for a bf16 layer, whose activations
    and per-pair rows are rounded to bf16; 3.9e-3 after four residual layers; 6e-7 in fp32; 7e-4 where only merged
    rows are rounded).  Selections are whole numbers: a token whose k-th and next expert tie within fp32 rounding may
    differ (seen: one of 5,488 and one of 60,000 slots)."""
    if case["shape"] == "tiny":
        return {"rel": 3e-6, "differ": 1e-3}
    if case["kind"] == "stage":
        return {"rel": 3e-3, "differ": 1e-3}
    return {"rel": 1.6e-2 if case["kind"] == "stack" else 1.2e-2, "differ": 1e-3}


# ---------------------------------------------------------------------------------------------- the same in 64 bits
def _from_fp8(q, e):
    G, R, C = q.shape
    v = q.view(torch.float8_e4m3fn).to(torch.float64).view(G, R // 128, 128, C // 128, 128)
    return (v * torch.exp2(e.to(torch.float64))[:, :, None, :, None]).reshape(G, R, C)


def _ffn64(x, gate, up, down):
    a = x @ gate.double().T
    return (a / (1.0 + torch.exp(-a)) * (x @ up.double().T)) @ down.double().T


def _layer64(case, w, x, mask, reduce_on, residual):
    s = _SHAPES[case["shape"]]
    K, Kv, E = s["top_k"], s["top_k_vis"], s["experts"]
    z = x @ w["router_w"].double().T
    if w["router_b"] is not None:
        z = z + w["router_b"].double()
    probs = torch.softmax(z, dim=1)
    top, idx = torch.topk(probs, K, dim=1)
    k = torch.full((x.shape[0], 1), K, device=x.device)
    if reduce_on:
        k[mask.bool()] = Kv
    top = torch.where(torch.arange(K, device=x.device)[None, :] < k, top, torch.zeros_like(top))
    gate = torch.zeros_like(probs).scatter_(1, idx, top / top.sum(dim=1, keepdim=True))
    out = x.clone() if residual else torch.zeros_like(x)

    def expert(name, i):
        m = w[name][i:i + 1]
        return (_from_fp8(m, w[name + "_scale"][i:i + 1]) if case["fp8"] else m)[0]

    for e in range(E):
        rows = torch.nonzero(gate[:, e] > 0)[:, 0]
        if rows.numel():
            y = _ffn64(x[rows], expert("w_gate", e), expert("w_up", e), expert("w_down", e))
            out.index_add_(0, rows, gate[rows, e, None] * y)
    for i in range(s["n_shared"]):
        out += _ffn64(x, expert("ws_gate", i), expert("ws_up", i), expert("ws_down", i))
    return out, probs


def _prune64(case, x, probs, attn, n_vis, off):
    W, rows = case["window"], []
    for b, (v, eta) in enumerate(zip(n_vis, _retain(case, n_vis))):
        lo = off[b]
        n_f = v // W
        kept, m = _kept(case, v, eta)
        d = (v - kept - m * (W - 1)) // W
        action = torch.zeros(n_f, dtype=torch.int64)
        if n_f:
            p = probs[lo:lo + n_f * W].view(n_f, W, -1)
            p = p / p.norm(dim=2, keepdim=True)
            gram = p @ p.transpose(1, 2)
            sim = (gram.sum(dim=(1, 2)) - gram.diagonal(dim1=1, dim2=2).sum(dim=1)) / (W * (W - 1))
            score, imp = sim, None
            if attn is not None:
                imp = attn[lo:lo + n_f * W].view(n_f, W).sum(dim=1)
                imp = imp / imp.max()
                score = case["alpha"] * sim - (1.0 - case["alpha"]) * imp
            by = torch.argsort(score.float(), descending=True, stable=True).cpu()
            action[by[:m]] = 1
            rest = by[m:] if imp is None else torch.argsort(imp.float(), stable=True).cpu()
            action[rest[action[rest] == 0][:d]] = 2
        seq = x[lo:off[b + 1]]
        win = seq[:n_f * W].view(n_f, W, -1)
        mean = win.mean(dim=1)
        merged = mean * (win.norm(dim=2).amax(dim=1) / mean.norm(dim=1))[:, None] if n_f else mean
        out = seq.clone()
        keep = torch.ones(seq.shape[0], dtype=torch.bool)
        for i in range(n_f):
            if action[i] == 1:
                out[i * W] = merged[i]
                keep[i * W + 1:(i + 1) * W] = False
            elif action[i] == 2:
                keep[i * W:(i + 1) * W] = False
        rows.append(out[keep.to(out.device)])
    return torch.cat(rows)


def exact(case, seed):
    d = _inputs(case, seed)
    n_vis, off = _layout(case)
    x = d["x"].double()
    none = {"keep_idx": None, "kind": None, "is_visual_out": None}
    if case["kind"] == "stage":
        attn = torch.empty(off[-1], dtype=torch.float64, device="cuda")
        k = d["k"].double().repeat_interleave(_HEADS // _KV_HEADS, dim=1)
        for b in range(case["batch"]):
            z = torch.einsum("thd,hd->ht", k[off[b]:off[b + 1]], d["q"][b].double()) / math.sqrt(_HEAD_DIM)
            attn[off[b]:off[b + 1]] = torch.softmax(z, dim=1).mean(dim=0)
        return {"attn": attn, "x_out": _prune64(case, x, d["probs"].double(), attn, n_vis, off), **none}
    if case["kind"] == "stack":
        for layer, w in enumerate(d["w"]):
            x, _ = _layer64(case, w, x, d["mask"], layer >= 1, True)
        return {"x_out": x, "is_visual_out": None}
    out, probs = _layer64(case, d["w"][0], x, d["mask"], True, case["residual"])
    if case["kind"] == "layer":
        return {"out": out}
    attn = None if d["attn"] is None else d["attn"].double()
    return {"out": out, "probs": probs, "topk_idx": None, "x_out": _prune64(case, out, probs, attn, n_vis, off), **none}

"""GPU parity: the whole MoE layer (Eq. 1-5) through the C ABI against the CPU oracle.
Tolerances: fp32 layers 1e-4, bf16 layers 2e-2, both as max over token rows of
|y - ref|_inf / |ref|_inf.  The oracle is teacher-forced on the kernel's fp32 logits for
the (integer) selection, so a near-tie cannot turn into a large output difference."""
import numpy as np
import pytest
import torch

from oracle import fmmoe_oracle as O
from paper_2511_17885_b200 import binding as B
from paper_2511_17885_b200 import inputs as I
from paper_2511_17885_b200.workload import upload_weights_fp8
from gpu_util import dev, handle, host, row_rel_err, upload_weights, TDT

pytestmark = pytest.mark.gpu
TOL = {"f32": 1e-4, "bf16": 2e-2}


def random_layer(r, dtype, H, E, I_, Ns, Is, std=0.05):
    def d(shape):
        return I.round_to_storage(std * r.standard_normal(shape), dtype)
    w = {"router_w": d((E, H)), "router_b": None, "w_gate": d((E, I_, H)), "w_up": d((E, I_, H)),
         "w_down": d((E, H, I_)), "ws_gate": None, "ws_up": None, "ws_down": None}
    if Ns:
        w["ws_gate"] = d((Ns, Is, H)); w["ws_up"] = d((Ns, Is, H)); w["ws_down"] = d((Ns, H, Is))
    return w


def run_layer(dtype, x, mask, w, K, Kv, flags, Ns=0, Is=0):
    td = TDT[dtype]
    T, H = x.shape
    E, I_ = w["w_gate"].shape[0], w["w_gate"].shape[1]
    desc = B.make_desc(H, E, I_, Ns, Is, K, Kv, td)
    wd = upload_weights(w, dtype)
    ws = B.make_weights(wd)
    route = {"logits": torch.empty(T, E, dtype=torch.float32, device="cuda"),
             "topk_idx": torch.empty(T, K, dtype=torch.int32, device="cuda"),
             "topk_w": torch.empty(T, K, dtype=torch.float32, device="cuda")}
    out = handle().fmmoe_moe_forward(desc, ws, dev(x, td), dev(mask), flags, route=route)
    handle().check_status()
    return host(out), {k: host(v) for k, v in route.items()}


def check_layer(dtype, T, H, E, I_, K, Kv, Ns=0, Is=0, flags=B.FLAG_REDUCE_ON, seed=0, mask=None, bias=False):
    r = np.random.default_rng(seed)
    x = I.round_to_storage(r.standard_normal((T, H)), dtype)
    mask = (r.random(T) < 0.7).astype(np.uint8) if mask is None else mask
    w = random_layer(r, dtype, H, E, I_, Ns, Is)
    if bias:
        w["router_b"] = (0.7 * r.standard_normal(E)).astype(np.float32)
    y, route = run_layer(dtype, x, mask, w, K, Kv, flags, Ns, Is)
    ref = O.moe_forward(x, mask, w, K, Kv, bool(flags & B.FLAG_REDUCE_ON), bool(flags & B.FLAG_RESIDUAL),
                        logits32=route["logits"])
    assert np.array_equal(route["topk_idx"], ref["topk_idx"])
    err = row_rel_err(y, ref["out"])
    assert err < TOL[dtype], f"row-relative error {err}"
    return y, ref


SMALL = [
    # dtype, T, H, E, I, K, Kv, Ns, Is
    ("f32", 256, 256, 8, 512, 2, 1, 0, 0),
    ("f32", 70, 64, 5, 36, 3, 1, 1, 20),
    ("bf16", 300, 128, 8, 128, 2, 1, 0, 0),
    ("bf16", 1000, 256, 16, 192, 4, 2, 2, 192),
    ("bf16", 515, 512, 40, 320, 6, 3, 1, 128),
    ("bf16", 129, 64, 4, 64, 2, 0, 1, 64),
]


@pytest.mark.parametrize("case", SMALL)
@pytest.mark.parametrize("det", [0, B.FLAG_DETERMINISTIC])
def test_layer_small(case, det):
    dtype, T, H, E, I_, K, Kv, Ns, Is = case
    check_layer(dtype, T, H, E, I_, K, Kv, Ns, Is, flags=B.FLAG_REDUCE_ON | det)


def test_layer_residual_and_reduce_off():
    check_layer("bf16", 200, 128, 8, 128, 3, 1, flags=B.FLAG_REDUCE_ON | B.FLAG_RESIDUAL)
    check_layer("bf16", 200, 128, 8, 128, 3, 1, flags=0)
    check_layer("f32", 90, 64, 6, 64, 2, 1, flags=B.FLAG_RESIDUAL)


def test_layer_edge_masks_and_empty_experts():
    T = 260
    check_layer("bf16", T, 128, 8, 128, 2, 1, mask=np.ones(T, np.uint8))
    check_layer("bf16", T, 128, 8, 128, 2, 1, mask=np.zeros(T, np.uint8))
    # a strong bias empties several experts and overloads others (multi-tile groups)
    r = np.random.default_rng(3)
    x = I.round_to_storage(r.standard_normal((T, 128)), "bf16")
    w = random_layer(r, "bf16", 128, 16, 128, 0, 0)
    w["router_b"] = np.array([8, 8, 8] + [-30] * 13, np.float32)
    mask = (r.random(T) < 0.5).astype(np.uint8)
    y, route = run_layer("bf16", x, mask, w, 3, 1, B.FLAG_REDUCE_ON)
    ref = O.moe_forward(x, mask, w, 3, 1, True, logits32=route["logits"])
    assert set(np.unique(route["topk_idx"][route["topk_idx"] >= 0]).tolist()) <= {0, 1, 2}
    assert row_rel_err(y, ref["out"]) < 2e-2


def test_layer_kv_equals_k_reproduces_dense():
    r = np.random.default_rng(4)
    T, H, E, I_ = 150, 128, 8, 128
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    mask = (r.random(T) < 0.6).astype(np.uint8)
    w = random_layer(r, "bf16", H, E, I_, 0, 0)
    a, _ = run_layer("bf16", x, mask, w, 3, 3, B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC)
    b, _ = run_layer("bf16", x, mask, w, 3, 1, B.FLAG_DETERMINISTIC)      # reduce off: K for everyone
    assert np.array_equal(a, b)


def test_layer_deterministic_mode_is_reproducible():
    r = np.random.default_rng(6)
    T, H, E, I_ = 400, 256, 16, 128
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    mask = (r.random(T) < 0.6).astype(np.uint8)
    w = random_layer(r, "bf16", H, E, I_, 1, 128)
    a, _ = run_layer("bf16", x, mask, w, 4, 2, B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC, 1, 128)
    b, _ = run_layer("bf16", x, mask, w, 4, 2, B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC, 1, 128)
    assert np.array_equal(a, b)


def test_layer_c0_full_config():
    cfg = I.C0
    x, m, _, _ = I.make_tokens(cfg)
    w = I.make_weights(cfg)
    y, route = run_layer("f32", x, m, w, cfg.top_k, cfg.top_k_vis, B.FLAG_REDUCE_ON)
    ref = O.moe_forward(x, m, w, cfg.top_k, cfg.top_k_vis, True, logits32=route["logits"])
    assert np.array_equal(route["topk_idx"], ref["topk_idx"])
    assert row_rel_err(y, ref["out"]) < 1e-4
    assert int((ref["topk_idx"] >= 0).sum()) == 224 * 1 + 32 * 2


def test_forward_host_variant_and_empty():
    r = np.random.default_rng(7)
    T, H, E, I_ = 200, 128, 8, 128
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    mask = (r.random(T) < 0.6).astype(np.uint8)
    w = random_layer(r, "bf16", H, E, I_, 0, 0)
    desc = B.make_desc(H, E, I_, 0, 0, 2, 1, torch.bfloat16)
    wd = upload_weights(w, "bf16"); ws = B.make_weights(wd)
    xh = torch.from_numpy(x).to(torch.bfloat16).pin_memory()
    mh = torch.from_numpy(mask).pin_memory()
    oh = torch.empty_like(xh).pin_memory()
    handle().fmmoe_moe_forward_host(desc, ws, xh, mh, B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC, oh)
    y, _ = run_layer("bf16", x, mask, w, 2, 1, B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC)
    assert np.array_equal(oh.float().numpy(), y)
    # T = 0
    out = handle().fmmoe_moe_forward(desc, ws, torch.zeros(0, H, dtype=torch.bfloat16, device="cuda"),
                                     torch.zeros(0, dtype=torch.uint8, device="cuda"), 1)
    assert out.shape == (0, H)


def test_pipelined_host_batches_match_the_device_path():
    """Five different batches through the pipelined host-buffer calls, two in flight: each batch's layer
    output and pruned rows (downloaded on the library's copy stream) equal the device-resident path's."""
    r = np.random.default_rng(11)
    T, H, E, I_, K, Kv = 300, 128, 8, 128, 2, 1
    w = random_layer(r, "bf16", H, E, I_, 0, 0)
    wd = upload_weights(w, "bf16"); ws = B.make_weights(wd)
    desc = B.make_desc(H, E, I_, 0, 0, K, Kv, torch.bfloat16)
    hd = handle()
    seq_off, n_vis = [0, T], [200]
    pp = B.prune_params(5, 0.05)
    n_ret = [100]
    route = {"probs": torch.empty(T, E, dtype=torch.float32, device="cuda")}
    xs = [torch.from_numpy(I.round_to_storage(r.standard_normal((T, H)), "bf16")).to(torch.bfloat16).pin_memory()
          for _ in range(5)]
    mask_np = np.zeros(T, np.uint8); mask_np[:200] = 1
    mask_h = torch.from_numpy(mask_np).pin_memory()
    slots = [{"out_dev": torch.empty(T, H, dtype=torch.bfloat16, device="cuda"),
              "mask_dev": torch.empty(T, dtype=torch.uint8, device="cuda"), "ticket": None} for _ in range(2)]
    got = []
    for i, xh in enumerate(xs):
        sl = slots[i % 2]
        if sl["ticket"] is not None:
            hd.fmmoe_host_wait(sl["ticket"])
        out_h = torch.empty(T, H, dtype=torch.bfloat16).pin_memory()
        hd.fmmoe_moe_forward_host_async(desc, ws, xh, mask_h, B.FLAG_REDUCE_ON, out_h, slot=i % 2, route=route,
                                        out_dev=sl["out_dev"], is_visual_dev=sl["mask_dev"])
        pr = hd.fmmoe_prune_visual(pp, route["probs"], None, sl["out_dev"], sl["mask_dev"], seq_off, n_vis, n_ret,
                                   want_aux=False)
        pr_h = torch.empty(pr["x_out"].shape, dtype=torch.bfloat16).pin_memory()
        hd.fmmoe_download_async(pr_h, pr["x_out"])
        sl["keep"] = pr["x_out"]
        sl["ticket"] = hd.fmmoe_host_fence()
        got.append((out_h, pr_h, sl["ticket"]))
    for out_h, pr_h, t in got:
        hd.fmmoe_host_wait(t)
    hd.check_status()
    mask_d = dev(mask_np)
    for xh, (out_h, pr_h, _) in zip(xs, got):
        ref = hd.fmmoe_moe_forward(desc, ws, xh.cuda(), mask_d, B.FLAG_REDUCE_ON, route=route)
        pr = hd.fmmoe_prune_visual(pp, route["probs"], None, ref, mask_d, seq_off, n_vis, n_ret, want_aux=False)
        # the combine adds in a different order from call to call (atomics): compare within the bf16 tolerance
        assert row_rel_err(out_h.float().numpy(), ref.float().cpu().numpy()) < 2e-2
        assert pr_h.shape == pr["x_out"].shape
        assert row_rel_err(pr_h.float().numpy(), pr["x_out"].float().cpu().numpy()) < 2e-2
    with pytest.raises(B.FmmoeError):
        hd.fmmoe_host_wait(1 << 40)


@pytest.mark.parametrize("use_attn", [False, True])
def test_layer_and_pruning_in_one_call_equals_the_two_calls(use_attn):
    """fmmoe_moe_forward_prune (selection on a side stream beside the GEMMs) against fmmoe_moe_forward followed by
    fmmoe_prune_visual: the same keep-set bit for bit; with the fixed-order combine also the same rows bit for bit."""
    r = np.random.default_rng(21)
    H, E, I_, K, Kv = 128, 16, 128, 4, 2
    seq_off, n_vis = [0, 700, 1030, 1500], [520, 200, 331]
    T = seq_off[-1]
    mask_np = np.zeros(T, np.uint8)
    for b in range(3):
        idx = r.permutation(seq_off[b + 1] - seq_off[b])[:n_vis[b]] + seq_off[b]   # vision tokens interleaved with text
        mask_np[idx] = 1
    n_ret = [260, 50, 331]
    w = random_layer(r, "bf16", H, E, I_, 1, 64)
    wd = upload_weights(w, "bf16"); ws = B.make_weights(wd)
    desc = B.make_desc(H, E, I_, 1, 64, K, Kv, torch.bfloat16)
    x = dev(I.round_to_storage(r.standard_normal((T, H)), "bf16"), torch.bfloat16)
    mask = dev(mask_np)
    attn = dev(r.random(T).astype(np.float32)) if use_attn else None
    pp = B.prune_params(3, 0.1, 0.6 if use_attn else 1.0)
    hd = handle()
    for flags in (B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC, B.FLAG_REDUCE_ON | B.FLAG_RESIDUAL):
        route_a = {"probs": torch.empty(T, E, dtype=torch.float32, device="cuda")}
        route_b = {"probs": torch.empty(T, E, dtype=torch.float32, device="cuda")}
        out_a = hd.fmmoe_moe_forward(desc, ws, x, mask, flags, route=route_a)
        ref = hd.fmmoe_prune_visual(pp, route_a["probs"], attn, out_a, mask, seq_off, n_vis, n_ret)
        out_b = torch.empty_like(x)
        for _ in range(2):   # twice: the side stream's second use must be ordered after the first
            got = hd.fmmoe_moe_forward_prune(desc, ws, x, mask, flags, out_b, route_b, pp, attn, seq_off, n_vis, n_ret)
        hd.check_status()
        assert got["out_seq_off"] == ref["out_seq_off"]
        assert torch.equal(route_a["probs"], route_b["probs"])
        for k in ("keep_idx", "kind", "is_visual_out"):
            assert torch.equal(got[k], ref[k]), k
        if flags & B.FLAG_DETERMINISTIC:
            assert torch.equal(out_a, out_b) and torch.equal(got["x_out"], ref["x_out"])
        else:
            assert row_rel_err(host(got["x_out"]), host(ref["x_out"])) < 2e-2
        # within one call the pruned rows are the call's own layer output: copied rows bit for bit
        copied = got["kind"] != 2
        assert torch.equal(got["x_out"][copied], out_b[got["keep_idx"][copied].long()])
    # argument errors surface before anything is enqueued
    with pytest.raises(B.FmmoeError):
        hd.fmmoe_moe_forward_prune(desc, ws, x, mask, B.FLAG_REDUCE_ON, out_b, route_b, pp, attn, [0, 700, 1030, 1499],
                                   n_vis, n_ret)


@pytest.mark.parametrize("H,K,W,lens,merge_mode,residual,in_place", [
    (2048, 8, 5, [611, 75], 0, False, False),       # the finalize pass writes the pruned rows: widest row it does
    (64, 16, 8, [300], 1, True, False), (192, 3, 2, [65, 0, 130], 0, True, False), (128, 1, 3, [64] * 64, 2, False, False),
    (2112, 2, 3, [280], 0, False, False),           # wider rows, more sequences, or the pruned rows over the layer's
    (128, 2, 3, [40] * 70, 0, False, False), (256, 4, 3, [300, 90], 0, True, True)])    # input: by the gather pass
def test_layer_and_pruning_in_one_call_on_both_routes_of_the_rows(H, K, W, lens, merge_mode, residual, in_place):
    """Both ways the single call produces the pruned rows give, bit for bit, the rows of the two separate calls (the same
    sums in the same order), K = 1 and 16, window sizes 2 and 8, short and empty sequences included.  Where the finalize
    pass writes them the call has one launch less than the two."""
    r = np.random.default_rng(H + K)
    T, E, I_ = sum(lens), 16, 64
    seq_off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    mask_np = (r.random(T) < 0.8).astype(np.uint8)
    n_vis = [int(mask_np[seq_off[b]:seq_off[b + 1]].sum()) for b in range(len(lens))]
    n_ret = [v // 2 for v in n_vis]
    w = random_layer(r, "bf16", H, E, I_, 1, 64)
    wd = upload_weights(w, "bf16"); ws = B.make_weights(wd)
    desc = B.make_desc(H, E, I_, 1, 64, K, max(K // 2, 1), torch.bfloat16)
    x = dev(I.round_to_storage(r.standard_normal((T, H)), "bf16"), torch.bfloat16)
    mask = dev(mask_np)
    pp = B.prune_params(W, 0.15, 1.0, 0, merge_mode)
    flags = B.FLAG_REDUCE_ON | (B.FLAG_RESIDUAL if residual else 0)
    hd = handle()
    route = {"probs": torch.empty(T, E, dtype=torch.float32, device="cuda")}
    n0 = hd.launch_count()
    out = hd.fmmoe_moe_forward(desc, ws, x, mask, flags, route=route)
    ref = hd.fmmoe_prune_visual(pp, route["probs"], None, out, mask, seq_off, n_vis, n_ret)
    n1 = hd.launch_count()
    out_b = torch.empty_like(x)
    if in_place:
        call = hd.prepare_forward_prune(desc, ws, x, mask, flags, out_b, route, pp, None, seq_off, n_vis, n_ret)
        args = list(call.args)
        args[15] = B._ptr(x)                        # x_out: the rows take the place of the layer's input, as in a stack
        assert call.fn(*args, B._stream()) == 0
        got = dict(call.result, x_out=x[:ref["x_out"].shape[0]])
    else:
        got = hd.fmmoe_moe_forward_prune(desc, ws, x, mask, flags, out_b, route, pp, None, seq_off, n_vis, n_ret)
    by_finalize = H <= 2048 and len(lens) <= 64 and not in_place
    assert hd.launch_count() - n1 == n1 - n0 - by_finalize
    hd.check_status()
    assert torch.equal(out, out_b)
    for k in ("keep_idx", "kind", "is_visual_out", "x_out"):
        assert torch.equal(got[k], ref[k]), k
    assert merge_mode == 2 or bool((got["kind"] == 2).any())


def test_layer_and_pruning_in_one_call_with_the_mask_compacted_in_place():
    """is_visual_out over is_visual in the single call: the outputs of the two separate calls, the mask where the old one was."""
    r = np.random.default_rng(57)
    lens, H, E = [400, 333, 90], 128, 16
    T = sum(lens)
    seq_off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    mask_np = (r.random(T) < 0.8).astype(np.uint8)
    n_vis = [int(mask_np[seq_off[b]:seq_off[b + 1]].sum()) for b in range(len(lens))]
    n_ret = [v // 2 for v in n_vis]
    wd = upload_weights(random_layer(r, "bf16", H, E, 64, 1, 64), "bf16"); ws = B.make_weights(wd)
    desc = B.make_desc(H, E, 64, 1, 64, 4, 2, torch.bfloat16)
    x = dev(I.round_to_storage(r.standard_normal((T, H)), "bf16"), torch.bfloat16)
    mask = dev(mask_np)
    pp = B.prune_params(3, 0.15, 1.0)
    hd = handle()
    route = {"probs": torch.empty(T, E, dtype=torch.float32, device="cuda")}
    out, out_b = torch.empty_like(x), torch.empty_like(x)
    ref = hd.fmmoe_moe_forward_prune(desc, ws, x, mask, B.FLAG_REDUCE_ON, out, route, pp, None, seq_off, n_vis, n_ret)
    call = hd.prepare_forward_prune(desc, ws, x, mask, B.FLAG_REDUCE_ON, out_b, route, pp, None, seq_off, n_vis, n_ret)
    args = list(call.args)
    args[16] = B._ptr(mask)                         # is_visual_out
    assert call.fn(*args, B._stream()) == 0
    hd.check_status()
    assert torch.equal(out, out_b)
    for k in ("keep_idx", "kind", "x_out"):
        assert torch.equal(call.result[k], ref[k]), k
    assert torch.equal(mask[:ref["is_visual_out"].numel()], ref["is_visual_out"])


def test_upload_and_download_streams_order_against_the_compute_stream():
    """fmmoe_upload_async -> device call -> fmmoe_download_async, four batches over two buffer sets."""
    r = np.random.default_rng(31)
    T, H, E, I_, K, Kv = 260, 128, 8, 128, 2, 1
    w = random_layer(r, "bf16", H, E, I_, 0, 0)
    wd = upload_weights(w, "bf16"); ws = B.make_weights(wd)
    desc = B.make_desc(H, E, I_, 0, 0, K, Kv, torch.bfloat16)
    hd = handle()
    mask = dev((r.random(T) < 0.6).astype(np.uint8))
    xs = [torch.from_numpy(I.round_to_storage(r.standard_normal((T, H)), "bf16")).to(torch.bfloat16).pin_memory()
          for _ in range(4)]
    sets = [{"x": torch.empty(T, H, dtype=torch.bfloat16, device="cuda"),
             "out": torch.empty(T, H, dtype=torch.bfloat16, device="cuda"), "ticket": None} for _ in range(2)]
    res = []
    for i, xh in enumerate(xs):
        st = sets[i % 2]
        if st["ticket"] is not None:
            hd.fmmoe_host_wait(st["ticket"])
        hd.fmmoe_upload_async(st["x"], xh)
        hd.fmmoe_moe_forward(desc, ws, st["x"], mask, B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC, out=st["out"])
        oh = torch.empty(T, H, dtype=torch.bfloat16).pin_memory()
        hd.fmmoe_download_async(oh, st["out"])
        st["ticket"] = hd.fmmoe_host_fence()
        res.append((oh, st["ticket"]))
    for oh, t in res:
        hd.fmmoe_host_wait(t)
    hd.check_status()
    for xh, (oh, _) in zip(xs, res):
        ref = hd.fmmoe_moe_forward(desc, ws, xh.cuda(), mask, B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC)
        assert torch.equal(oh, ref.cpu())


def test_host_tickets_survive_the_ring_wrapping_around():
    """More fences than the handle keeps events for: every ticket, however old, can still be waited for."""
    hd = handle()
    src = torch.arange(1024, dtype=torch.int32, device="cuda")
    dst = torch.zeros(1024, dtype=torch.int32).pin_memory()
    tickets = []
    for i in range(150):
        src.add_(1)
        hd.fmmoe_download_async(dst, src)
        tickets.append(hd.fmmoe_host_fence())
    assert tickets == list(range(tickets[0], tickets[0] + 150))
    for t in (tickets[0], tickets[70], tickets[-1]):
        hd.fmmoe_host_wait(t)
    assert torch.equal(dst, src.cpu())
    with pytest.raises(B.FmmoeError):
        hd.fmmoe_host_wait(tickets[-1] + 1)


def _rows_per_expert_case(counts, n_text_extra, H=128, I_=192, seed=41):
    """Tokens whose first choice is fixed by construction, so that expert e receives exactly counts[e] first-choice
    rows: vision tokens (K_v = 1) carry their whole weight on that expert.  `n_text_extra` text tokens (K = 2) all
    take the last two experts, which therefore hold several M-tiles."""
    r = np.random.default_rng(seed)
    E = len(counts) + 2
    assign = np.concatenate([np.full(c, e) for e, c in enumerate(counts)]).astype(np.int64)
    r.shuffle(assign)
    T = assign.size + n_text_extra
    x = 0.25 * r.standard_normal((T, H))
    mask = np.ones(T, np.uint8)
    mask[assign.size:] = 0
    w = random_layer(r, "bf16", H, E, I_, 0, 0)
    router = np.zeros((E, H))
    for e in range(E):
        router[e, e] = 1.0                      # logit of expert e = x[t, e]
    w["router_w"] = I.round_to_storage(router, "bf16")
    x[np.arange(assign.size), assign] = 8.0     # first choice of every vision token
    x[assign.size:, E - 2] = 8.0                # text tokens: the two big experts
    x[assign.size:, E - 1] = 6.0
    return I.round_to_storage(x, "bf16"), mask, w, E


_ATOMIC = {"FMMOE_PAIR_ROWS_MIN_TOKENS": "1000000"}       # the atomic fp32 combine (optional; the default is pair rows)
ROW_PATHS = {
    # name: environment read by fmmoe_create -> which kernels the expert GEMMs run as at this size
    # one CTA a tile of up to 128 rows, and CTA pairs with tiles of up to 256, at every size; two names of one threshold
    "small_m": dict({"FMMOE_SMALL_M_MAX_TOKENS": "1000000"}, **_ATOMIC),
    "cta_pairs": dict({"FMMOE_SMALL_M_MAX_TOKENS": "0"}, **_ATOMIC),
    # the combine through per-pair bf16 rows (the default), under both forms
    "small_m_pair_rows": {"FMMOE_CTA_PAIR_MIN_TOKENS": "1000000"},
    "cta_pairs_pair_rows": {"FMMOE_CTA_PAIR_MIN_TOKENS": "0"},
}


def handle_with_env(monkeypatch, env):
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    h = B.Handle(0)                                  # the thresholds are read once, when the handle is created
    for k in env:
        monkeypatch.delenv(k, raising=False)
    return h


@pytest.mark.parametrize("path", list(ROW_PATHS))
def test_rows_per_expert_boundaries_on_every_gemm_form(path, monkeypatch):
    """Experts holding 0, 1, 15, 16, 17, 33, 64, 65, 96, 97, 128 and 129 rows (and two with several hundred), EVERY
    output row against the oracle, on both forms of the expert GEMMs with both combines."""
    counts = [0, 1, 15, 16, 17, 33, 64, 65, 96, 97, 128, 129]
    x, mask, w, E = _rows_per_expert_case(counts, n_text_extra=300)
    h = handle_with_env(monkeypatch, ROW_PATHS[path])
    T, H = x.shape
    I_ = w["w_gate"].shape[1]
    desc = B.make_desc(H, E, I_, 0, 0, 2, 1, torch.bfloat16)
    assert h.fmmoe_test_gemm_form(desc, T) == (2 if "pairs" in path else 1)
    wd = upload_weights(w, "bf16"); ws = B.make_weights(wd)
    route = {"logits": torch.empty(T, E, dtype=torch.float32, device="cuda"),
             "topk_idx": torch.empty(T, 2, dtype=torch.int32, device="cuda"),
             "expert_off": torch.empty(E + 1, dtype=torch.int32, device="cuda")}
    for flags in (B.FLAG_REDUCE_ON, B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC):
        out = h.fmmoe_moe_forward(desc, ws, dev(x, torch.bfloat16), dev(mask), flags, route=route)
        h.check_status()
        got_counts = np.diff(host(route["expert_off"]))
        assert got_counts[:len(counts)].tolist() == counts and got_counts[-1] == 300 and got_counts[-2] == 300
        ref = O.moe_forward(x, mask, w, 2, 1, True, logits32=host(route["logits"]))
        assert np.array_equal(host(route["topk_idx"]), ref["topk_idx"])
        assert row_rel_err(host(out), ref["out"]) < 2e-2
    h.close()


@pytest.mark.parametrize("T,H,E,I_,K,Kv,Ns,Is", [
    (1, 4, 1, 4, 1, 1, 0, 0), (33, 132, 3, 68, 2, 1, 1, 36), (96, 60, 7, 100, 3, 2, 0, 0), (64, 516, 40, 132, 4, 2, 0, 0),
    (40, 128, 250, 32, 5, 3, 2, 128)])
def test_fp32_layer_at_the_edges_of_its_tiles_and_slabs(T, H, E, I_, K, Kv, Ns, Is):
    """fp32 layers whose contraction lengths are below, at and just past a slab (64 for the router, 128 for the expert
    GEMMs), whose widths leave partial 32- and 64-row blocks, and with 1 and 250 experts; both combines."""
    for flags in (B.FLAG_REDUCE_ON, B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC | B.FLAG_RESIDUAL):
        check_layer("f32", T, H, E, I_, K, Kv, Ns, Is, flags=flags, seed=T + H)


@pytest.mark.parametrize("T", [1, 7, 16, 40])
def test_decode_sized_batches_with_shared_experts(T):
    """A handful of tokens (a decode step): every expert holds 0-3 rows, so each routed tile is one 16-row MMA
    column block; shared experts and odd feature-block counts (S_m = 192 = 128 + 64) included."""
    check_layer("bf16", T, 256, 16, 192, 4, 2, 1, 192, flags=B.FLAG_REDUCE_ON, seed=50 + T)
    check_layer("bf16", T, 128, 8, 64, 2, 1, 0, 0, flags=B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC, seed=60 + T)


@pytest.mark.parametrize("T,H,E,I_,K,Kv,Ns,Is", [
    (1, 2048, 8, 192, 4, 2, 1, 64),        # 5 M-tiles x 16 blocks: one round; 3 and 1 k-blocks
    (1, 2048, 16, 64, 9, 9, 0, 0),         # 144 tiles of 128 features
    (1, 2048, 16, 64, 10, 10, 0, 0),       # 160: blocks of 256
    (32, 320, 16, 320, 8, 4, 2, 128),      # 32 rows, a block of 64 features at the end
    (33, 320, 16, 320, 8, 4, 2, 128)])     # more rows than two boxes of a stage hold
def test_few_tiles_take_half_the_features_in_gemm2(T, H, E, I_, K, Kv, Ns, Is):
    """GEMM-2 tiles of 128 features, two k-blocks a stage: odd and even numbers of k-blocks, the last feature block
    partial, and both sides of the rule (all tiles in one round of the SMs, at most 32 tokens), in each combine."""
    for flags in (B.FLAG_REDUCE_ON | B.FLAG_RESIDUAL, B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC):
        check_layer("bf16", T, H, E, I_, K, Kv, Ns, Is, flags=flags, seed=T + K)


@pytest.mark.parametrize("T,H,E,I_,K,fp8,form", [
    (1023, 192, 64, 320, 8, False, 1), (1024, 192, 64, 320, 8, False, 2),      # an average of 128 rows per expert (64 x 3 tiles)
    (1279, 256, 64, 384, 8, True, 1), (1280, 256, 64, 384, 8, True, 2),        # 160 with FP8 weights
    (255, 64, 16, 1280, 16, False, 1), (256, 64, 16, 1280, 16, False, 2),      # 256 tokens (255 or 256 rows per expert, 16 x 10 tiles)
    (256, 64, 16, 1152, 16, False, 1)])                                        # 16 x 9 tiles leave SMs without one
def test_default_form_on_both_sides_of_its_rule(T, H, E, I_, K, fp8, form):
    """With the handle's defaults the expert GEMMs run on CTA pairs from certain numbers of rows, tokens and tiles on: a layer
    on either side of each, shared experts and residual included, against the oracle."""
    assert torch.cuda.get_device_properties(0).multi_processor_count == 148      # what the numbers of tiles stand against
    r = np.random.default_rng(300 + T)
    Is, Kv = 128, K // 2
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    mask = (r.random(T) < 0.7).astype(np.uint8)
    w = random_layer(r, "bf16", H, E, I_, 1, Is)
    if fp8:
        w, packed = I.weights_to_fp8(w)
        wd = upload_weights_fp8(w, packed, "bf16", "cuda")
    else:
        wd = upload_weights(w, "bf16")
    desc = B.make_desc(H, E, I_, 1, Is, K, Kv, torch.bfloat16, B.WEIGHTS_FP8_BLOCK128 if fp8 else B.WEIGHTS_AS_DTYPE)
    h = handle()
    assert h.fmmoe_test_gemm_form(desc, T) == form
    ws = B.make_weights(wd)
    route = {"logits": torch.empty(T, E, dtype=torch.float32, device="cuda")}
    out = h.fmmoe_moe_forward(desc, ws, dev(x, torch.bfloat16), dev(mask), B.FLAG_REDUCE_ON | B.FLAG_RESIDUAL, route=route)
    h.check_status()
    ref = O.moe_forward(x, mask, w, K, Kv, True, add_residual=True, logits32=host(route["logits"]))
    assert row_rel_err(host(out), ref["out"]) < 2e-2


def test_both_forms_agree_bit_for_bit_in_fixed_order_mode(monkeypatch):
    """The two forms of the expert GEMMs (one CTA a tile, CTA pairs) accumulate every output element over the same k order in
    fp32, so with the fixed-order combine their layer outputs are identical bit for bit."""
    r = np.random.default_rng(71)
    T, H, E, I_ = 900, 256, 16, 320
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    mask = (r.random(T) < 0.7).astype(np.uint8)
    w = random_layer(r, "bf16", H, E, I_, 1, 128)
    outs = []
    for form in ("small_m", "cta_pairs"):
        h = handle_with_env(monkeypatch, ROW_PATHS[form])
        desc = B.make_desc(H, E, I_, 1, 128, 4, 2, torch.bfloat16)
        wd = upload_weights(w, "bf16"); ws = B.make_weights(wd)
        outs.append(h.fmmoe_moe_forward(desc, ws, dev(x, torch.bfloat16), dev(mask),
                                        B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC).clone())
        h.check_status()
        h.close()
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("form", ["small_m_pair_rows", "cta_pairs_pair_rows"])
@pytest.mark.parametrize("k_block", [0, 5])
def test_bounded_wait_runs_out_and_the_handle_recovers(k_block, form, monkeypatch):
    """The producer of GEMM-1 (one CTA or one pair, tiny shape) stops before it issues k-block `k_block`; the issuing thread's
    wait for that stage has a 3 ms budget and nothing will ever complete it.  Expected: the call returns, the kernels
    finish, fmmoe_get_status reports FMMOE_ERR_TIMEOUT exactly once, and the next ordinary call on the same handle
    passes parity (tensor memory was released, no barrier is left half-way)."""
    h = handle_with_env(monkeypatch, ROW_PATHS[form])
    r = np.random.default_rng(81)
    T, H, E, I_ = 96, 512, 4, 128            # H = 512: eight k-blocks per GEMM-1 tile
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    mask = (r.random(T) < 0.5).astype(np.uint8)
    w = random_layer(r, "bf16", H, E, I_, 0, 0)
    desc = B.make_desc(H, E, I_, 0, 0, 2, 1, torch.bfloat16)
    wd = upload_weights(w, "bf16"); ws = B.make_weights(wd)
    xd, md = dev(x, torch.bfloat16), dev(mask)
    h.fmmoe_test_expire_wait(3_000_000, k_block)
    h.fmmoe_moe_forward(desc, ws, xd, md, B.FLAG_REDUCE_ON)
    assert h.get_status() == 5                # FMMOE_ERR_TIMEOUT, read and cleared
    assert h.get_status() == 0
    route = {"logits": torch.empty(T, E, dtype=torch.float32, device="cuda")}
    out = h.fmmoe_moe_forward(desc, ws, xd, md, B.FLAG_REDUCE_ON, route=route)
    h.check_status()
    ref = O.moe_forward(x, mask, w, 2, 1, True, logits32=host(route["logits"]))
    assert row_rel_err(host(out), ref["out"]) < 2e-2
    h.close()


@pytest.mark.parametrize("k_block,status", [(31, 5), (32, 0), (35, 0), (47, 0), (48, 0)])
def test_held_back_k_blocks_are_the_first_gemms(k_block, status, monkeypatch):
    """Four experts of one M-tile and one feature block each: GEMM-1 has 32 k-blocks, GEMM-2, in the same launch, sixteen more, none of which the
    self-test holds back."""
    h = handle_with_env(monkeypatch, ROW_PATHS["small_m_pair_rows"])
    r = np.random.default_rng(82)
    T, H, E, I_ = 96, 512, 4, 128
    w = random_layer(r, "bf16", H, E, I_, 0, 0)
    w["router_b"] = np.zeros(E, np.float32)
    desc = B.make_desc(H, E, I_, 0, 0, 4, 4, torch.bfloat16)       # every token takes every expert
    ws = B.make_weights(upload_weights(w, "bf16"))
    x, mask = dev(I.round_to_storage(r.standard_normal((T, H)), "bf16"), torch.bfloat16), torch.zeros(T, dtype=torch.uint8, device="cuda")
    want = h.fmmoe_moe_forward(desc, ws, x, mask, 0)
    h.check_status()
    h.fmmoe_test_expire_wait(20_000_000, k_block)
    out = h.fmmoe_moe_forward(desc, ws, x, mask, 0)
    assert h.get_status() == status and h.get_status() == 0
    assert status or torch.equal(out, want)
    h.close()


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("form", ["small_m_pair_rows", "cta_pairs_pair_rows"])
@pytest.mark.parametrize("budget_ns", [1_000, 5_000, 20_000, 100_000])
def test_waits_that_run_out_anywhere(budget_ns, form, fp8, monkeypatch):
    """Budgets about as long as the waits themselves: any of them may run out, in any role and at any tile, while others
    go on.  The call returns, the status says TIMEOUT if one did, and the next ordinary call is right."""
    h = handle_with_env(monkeypatch, ROW_PATHS[form])
    r = np.random.default_rng(83)
    T, H, E, I_, Ns, Is = 200, 512, 8, 256, 1, 128
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    mask = (r.random(T) < 0.5).astype(np.uint8)
    w = random_layer(r, "bf16", H, E, I_, Ns, Is)
    if fp8:
        w, packed = I.weights_to_fp8(w)
        wd = upload_weights_fp8(w, packed, "bf16", "cuda")
    else:
        wd = upload_weights(w, "bf16")
    desc = B.make_desc(H, E, I_, Ns, Is, 2, 1, torch.bfloat16, B.WEIGHTS_FP8_BLOCK128 if fp8 else B.WEIGHTS_AS_DTYPE)
    ws = B.make_weights(wd)
    xd, md = dev(x, torch.bfloat16), dev(mask)
    for _ in range(5):
        h.fmmoe_test_expire_wait(budget_ns, 1_000_000)          # no k-block is held back
        h.fmmoe_moe_forward(desc, ws, xd, md, B.FLAG_REDUCE_ON)
        assert h.get_status() in (0, 5)
    route = {"logits": torch.empty(T, E, dtype=torch.float32, device="cuda")}
    out = h.fmmoe_moe_forward(desc, ws, xd, md, B.FLAG_REDUCE_ON, route=route)
    h.check_status()
    ref = O.moe_forward(x, mask, w, 2, 1, True, logits32=host(route["logits"]))
    assert row_rel_err(host(out), ref["out"]) < 2e-2
    h.close()


@pytest.mark.parametrize("T", [700, 513, 543, 545])          # shared experts: a last tile of 188, 1, 31 and 33 rows (pairs)
@pytest.mark.parametrize("path", ["small_m_pair_rows", "cta_pairs_pair_rows", "cta_pairs"])
def test_pair_row_combine_with_shared_experts_residual_and_reproducibility(path, T, monkeypatch):
    """The combine through per-pair bf16 rows: shared experts, residual, K_v = 0 tokens, against the oracle within
    the bf16 tolerance; it sums in a fixed order without atomics, so two runs agree bit for bit."""
    h = handle_with_env(monkeypatch, ROW_PATHS[path])
    r = np.random.default_rng(91)
    H, E, I_, Ns, Is, K, Kv = 256, 16, 192, 2, 128, 4, 0
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    mask = (r.random(T) < 0.6).astype(np.uint8)
    w = random_layer(r, "bf16", H, E, I_, Ns, Is)
    desc = B.make_desc(H, E, I_, Ns, Is, K, Kv, torch.bfloat16)
    wd = upload_weights(w, "bf16"); ws = B.make_weights(wd)
    route = {"logits": torch.empty(T, E, dtype=torch.float32, device="cuda")}
    flags = B.FLAG_REDUCE_ON | B.FLAG_RESIDUAL
    a = h.fmmoe_moe_forward(desc, ws, dev(x, torch.bfloat16), dev(mask), flags, route=route).clone()
    b = h.fmmoe_moe_forward(desc, ws, dev(x, torch.bfloat16), dev(mask), flags, route=route)
    h.check_status()
    if "pair_rows" in path:          # the atomic combine adds in arrival order
        assert torch.equal(a, b)
    ref = O.moe_forward(x, mask, w, K, Kv, True, add_residual=True, logits32=host(route["logits"]))
    assert row_rel_err(host(a), ref["out"]) < 2e-2
    h.close()


@pytest.mark.parametrize("H,I_", [(128, 192), (320, 64)])
def test_pair_tiles_at_the_edges_of_their_rows_and_features(H, I_, monkeypatch):
    """CTA pairs: experts of 31 ... 33, 255 ... 257 and 513 rows (one, two and three tiles that share the rows in steps of 32),
    widths that leave the partner CTA half or no valid features in the last block, an odd number of k-blocks; every output row
    against the oracle, and the per-pair and the fixed-order combine."""
    counts = [31, 32, 33, 255, 256, 257, 513, 0, 1]
    x, mask, w, E = _rows_per_expert_case(counts, n_text_extra=40, H=H, I_=I_)
    h = handle_with_env(monkeypatch, ROW_PATHS["cta_pairs_pair_rows"])
    T = x.shape[0]
    desc = B.make_desc(H, E, I_, 0, 0, 2, 1, torch.bfloat16)
    ws = B.make_weights(upload_weights(w, "bf16"))
    route = {"logits": torch.empty(T, E, dtype=torch.float32, device="cuda")}
    for flags in (B.FLAG_REDUCE_ON, B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC):
        out = h.fmmoe_moe_forward(desc, ws, dev(x, torch.bfloat16), dev(mask), flags, route=route)
        h.check_status()
        ref = O.moe_forward(x, mask, w, 2, 1, True, logits32=host(route["logits"]))
        assert row_rel_err(host(out), ref["out"]) < 2e-2
    h.close()


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("T,H,E,I_,Ns,Is", [
    (40, 128, 4, 128, 0, 0),            # fewer tiles than pairs, two k-blocks each: most rings are never filled once
    (600, 1024, 8, 384, 1, 128),        # several tiles a pair, sixteen k-blocks
    (3000, 256, 16, 256, 2, 256)])      # more tiles than a pair's mailbox holds
def test_pairs_leave_nothing_under_way(T, H, E, I_, Ns, Is, fp8, monkeypatch):
    """A CTA of a pair leaves only after everything that its partner and the pair's MMAs signal to it has arrived: with
    FMMOE_DEBUG_SYNC=1 the kernel looks at its own barriers as it leaves and reports INTERNAL if a signal is missing."""
    h = handle_with_env(monkeypatch, {"FMMOE_CTA_PAIR_MIN_TOKENS": "0", "FMMOE_DEBUG_SYNC": "1"})
    r = np.random.default_rng(T)
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    mask = (r.random(T) < 0.6).astype(np.uint8)
    w = random_layer(r, "bf16", H, E, I_, Ns, Is)
    if fp8:
        w, packed = I.weights_to_fp8(w)
        wd = upload_weights_fp8(w, packed, "bf16", "cuda")
    else:
        wd = upload_weights(w, "bf16")
    desc = B.make_desc(H, E, I_, Ns, Is, 4, 2, torch.bfloat16, B.WEIGHTS_FP8_BLOCK128 if fp8 else B.WEIGHTS_AS_DTYPE)
    ws = B.make_weights(wd)
    xd, md = dev(x, torch.bfloat16), dev(mask)
    route = {"logits": torch.empty(T, E, dtype=torch.float32, device="cuda")}
    for _ in range(20):
        out = h.fmmoe_moe_forward(desc, ws, xd, md, B.FLAG_REDUCE_ON, route=route)
    h.check_status()
    ref = O.moe_forward(x, mask, w, 4, 2, True, logits32=host(route["logits"]))
    assert row_rel_err(host(out), ref["out"]) < 2e-2
    h.close()


@pytest.mark.parametrize("T,Ns,Is", [(3, 2, 128), (200, 1, 9472), (200, 1, 9600)])      # 2, 148 and 150 tiles of shared experts in GEMM-1
def test_shared_experts_start_on_the_layers_own_inputs(T, Ns, Is):
    """The small-M form works on shared experts while the router runs, on fewer, as many and more tiles than there are SMs.  Rows,
    weights and the mask are overwritten on the stream right in front of every call, which has to see them: each output against the oracle,
    and bit for bit what a call on buffers that were there before gives."""
    r = np.random.default_rng(T + Is)
    H, E, I_, K = 128, 8, 64, 2
    cases = []
    for _ in range(3):
        w = random_layer(r, "bf16", H, E, I_, Ns, Is)
        cases.append((I.round_to_storage(r.standard_normal((T, H)), "bf16"), (r.random(T) < 0.5).astype(np.uint8), w))
    desc = B.make_desc(H, E, I_, Ns, Is, K, 1, torch.bfloat16)
    hd = handle()
    staged = [(dev(x, torch.bfloat16), dev(m), upload_weights(w, "bf16")) for x, m, w in cases]
    want = [hd.fmmoe_moe_forward(desc, B.make_weights(w), x, m, B.FLAG_REDUCE_ON) for x, m, w in staged]
    x, m, w = torch.empty_like(staged[0][0]), torch.empty_like(staged[0][1]), {k: v if v is None else torch.empty_like(v) for k, v in staged[0][2].items()}
    ws, got = B.make_weights(w), []
    for xs, ms, wd in staged:
        x.copy_(xs); m.copy_(ms)
        for k, v in w.items():
            if v is not None:
                v.copy_(wd[k])
        got.append(hd.fmmoe_moe_forward(desc, ws, x, m, B.FLAG_REDUCE_ON))
    hd.check_status()
    for (xn, mn, wn), a, b in zip(cases, want, got):
        assert torch.equal(a, b)
        assert row_rel_err(host(b), O.moe_forward(xn, mn, wn, K, 1, True)["out"]) < 2e-2


def test_gemms_in_one_launch_equal_the_two_of_a_timed_run():
    """The small-M form does both GEMMs in one launch, and in two when kernels are timed one by one: the same output bit for bit, from a
    single GEMM-2 tile to several a CTA, shared experts behind and between the routed ones."""
    r = np.random.default_rng(141)
    for T, H, E, I_, K, Ns, Is in [(1, 128, 4, 64, 1, 0, 64), (1, 2048, 16, 192, 6, 2, 128), (40, 1024, 32, 320, 4, 1, 192), (700, 512, 48, 256, 4, 2, 128)]:
        w = random_layer(r, "bf16", H, E, I_, Ns, Is)
        x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
        mask = (r.random(T) < 0.5).astype(np.uint8)
        desc = B.make_desc(H, E, I_, Ns, Is if Ns else 0, K, 1, torch.bfloat16)
        hd = handle()
        assert hd.fmmoe_test_gemm_form(desc, T) == 1
        ws, xd, md = B.make_weights(upload_weights(w, "bf16")), dev(x, torch.bfloat16), dev(mask)
        n0 = hd.launch_count()
        outs = [hd.fmmoe_moe_forward(desc, ws, xd, md, B.FLAG_REDUCE_ON) for _ in range(5)]
        n1 = hd.launch_count()
        hd.profile_enable()
        want = hd.fmmoe_moe_forward(desc, ws, xd, md, B.FLAG_REDUCE_ON)
        hd.profile_enable(False)
        assert hd.launch_count() - n1 == (n1 - n0) // 5 + 1
        hd.check_status()
        assert all(torch.equal(want, o) for o in outs)
        assert row_rel_err(host(want), O.moe_forward(x, mask, w, K, 1, True)["out"]) < 2e-2


def test_layers_of_two_handles_at_once():
    """Two layers on two streams share the SMs, so that neither's CTAs all run at the same time: no CTA waits for one that does not."""
    r = np.random.default_rng(151)
    T, H, E, I_, K, Ns, Is = 300, 1024, 32, 256, 4, 1, 256
    w = random_layer(r, "bf16", H, E, I_, Ns, Is)
    desc = B.make_desc(H, E, I_, Ns, Is, K, 2, torch.bfloat16)
    ws = B.make_weights(upload_weights(w, "bf16"))
    mask = dev((r.random(T) < 0.5).astype(np.uint8))
    xs = [dev(I.round_to_storage(r.standard_normal((T, H)), "bf16"), torch.bfloat16) for _ in range(2)]
    hs, streams = [B.Handle(0), B.Handle(0)], [torch.cuda.Stream(), torch.cuda.Stream()]
    want = [hs[i].fmmoe_moe_forward(desc, ws, xs[i], mask, B.FLAG_REDUCE_ON) for i in range(2)]
    torch.cuda.synchronize()
    got = [[], []]
    for _ in range(50):
        for i in range(2):
            with torch.cuda.stream(streams[i]):
                got[i].append(hs[i].fmmoe_moe_forward(desc, ws, xs[i], mask, B.FLAG_REDUCE_ON))
    torch.cuda.synchronize()
    for i in range(2):
        hs[i].check_status()
        assert all(torch.equal(want[i], o) for o in got[i])
        hs[i].close()


@pytest.mark.parametrize("shift", [0, 8, -8, 200])
@pytest.mark.parametrize("residual", [0, B.FLAG_RESIDUAL])
def test_fp32_output_over_part_of_the_input(shift, residual):
    """An fp32 layer without the residual is summed up in the output buffer itself, unless that lies over rows the layer still reads.  With
    the residual, which is read while the output is written, such an output is refused."""
    r = np.random.default_rng(161)
    T, H, E, I_, K, Ns = 150, 64, 6, 300, 2, 1
    w = random_layer(r, "f32", H, E, I_, Ns, 132)
    x = r.standard_normal((T, H)).astype(np.float32)
    mask = (r.random(T) < 0.5).astype(np.uint8)
    desc = B.make_desc(H, E, I_, Ns, 132, K, 1, torch.float32)
    ws = B.make_weights(upload_weights(w, "f32"))
    buf = torch.zeros(T + 400, H, device="cuda")
    xd, out = buf[200:200 + T], buf[200 + shift:200 + shift + T]
    xd.copy_(dev(x))
    if shift == 0:
        out = torch.full_like(xd, 7.0)             # a buffer of its own, with something in it
    if residual and abs(shift) == 8:
        refused_over_the_input(desc, ws, xd, dev(mask), out)
        return
    handle().fmmoe_moe_forward(desc, ws, xd, dev(mask), B.FLAG_REDUCE_ON | residual, out=out)
    handle().check_status()
    ref = O.moe_forward(x, mask, w, K, 1, True, add_residual=bool(residual))
    assert row_rel_err(host(out), ref["out"]) < 1e-4


def refused_over_the_input(desc, ws, x, mask, out):
    """Nothing is launched and x is as it was."""
    before, n0 = x.clone(), handle().launch_count()
    with pytest.raises(B.FmmoeError) as e:
        handle().fmmoe_moe_forward(desc, ws, x, mask, B.FLAG_REDUCE_ON | B.FLAG_RESIDUAL, out=out)
    assert e.value.status == 1 and handle().launch_count() == n0 and torch.equal(before, x)


@pytest.mark.parametrize("T", [5, 300])
def test_bf16_output_over_part_of_the_input(T):
    """Without the residual x has been read when the first row of the output is written; with it such an output is refused, from one row
    that both have in common on."""
    r = np.random.default_rng(T)
    H, E, I_, K = 128, 8, 128, 2
    w = random_layer(r, "bf16", H, E, I_, 0, 64)
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    mask = (r.random(T) < 0.5).astype(np.uint8)
    desc = B.make_desc(H, E, I_, 0, 0, K, 1, torch.bfloat16)
    ws = B.make_weights(upload_weights(w, "bf16"))
    for shift in (1, 1 - T, T, -T):
        buf = torch.zeros(3 * T, H, dtype=torch.bfloat16, device="cuda")
        xd, out = buf[T:2 * T], buf[T + shift:2 * T + shift]
        xd.copy_(dev(x, torch.bfloat16))
        if abs(shift) < T:
            refused_over_the_input(desc, ws, xd, dev(mask), out)
            residual = 0
        else:
            residual = B.FLAG_RESIDUAL             # side by side
        handle().fmmoe_moe_forward(desc, ws, xd, dev(mask), B.FLAG_REDUCE_ON | residual, out=out)
        handle().check_status()
        ref = O.moe_forward(x, mask, w, K, 1, True, add_residual=bool(residual))
        assert row_rel_err(host(out), ref["out"]) < 2e-2


@pytest.mark.parametrize("n_vis,n_text,Ns,fp8,pairs", [
    (1752, 48, 0, False, False), (1760, 48, 0, False, True),      # 64 experts, top-8 and 4: 116 rows of an expert on
    (850, 80, 1, False, False), (1700, 280, 1, False, True), (1480, 90, 0, True, False), (1484, 92, 0, True, True)])      # shared ones count; FP8: 104
def test_form_by_the_rows_that_exist_where_the_host_knows_the_vision_tokens(n_vis, n_text, Ns, fp8, pairs):
    """A call with a pruning stage and a stack choose the form of the expert GEMMs by the rows that exist; the plain call counts top_k for
    every token.  Same output bit for bit; pairs launch their two GEMMs one by one."""
    r = np.random.default_rng(n_vis)
    T, H, E, I_, Is = n_vis + n_text, 256, 64, 384, 128
    rows = (n_vis * 4 + n_text * 8 + Ns * T) / (E + Ns)
    assert pairs == (rows >= (104 if fp8 else 116))
    w = random_layer(r, "bf16", H, E, I_, Ns, Is)
    if fp8:
        w, packed = I.weights_to_fp8(w)
        wd = upload_weights_fp8(w, packed, "bf16", "cuda")
    else:
        wd = upload_weights(w, "bf16")
    desc = B.make_desc(H, E, I_, Ns, Is if Ns else 0, 8, 4, torch.bfloat16, B.WEIGHTS_FP8_BLOCK128 if fp8 else B.WEIGHTS_AS_DTYPE)
    ws = B.make_weights(wd)
    x = dev(I.round_to_storage(r.standard_normal((T, H)), "bf16"), torch.bfloat16)
    mask = dev(np.concatenate([np.ones(n_vis, np.uint8), np.zeros(n_text, np.uint8)]))
    hd = handle()
    route = {"probs": torch.empty(T, E, dtype=torch.float32, device="cuda")}
    want = hd.fmmoe_moe_forward(desc, ws, x, mask, B.FLAG_REDUCE_ON)
    out = torch.empty_like(x)
    n0 = hd.launch_count()
    hd.fmmoe_moe_forward_prune(desc, ws, x, mask, B.FLAG_REDUCE_ON, out, route, B.prune_params(5, 0.05), None, [0, T], [n_vis], [n_vis // 2])
    n1 = hd.launch_count()
    y, _, _ = hd.fmmoe_stack_forward(desc, [ws], 0, [], x, mask, [0, T], [n_vis])
    n2 = hd.launch_count()
    hd.check_status()
    assert n1 - n0 == 6 + pairs and n2 - n1 == 4 + pairs      # router, permutation, GEMMs, finalize; scores and selection
    assert torch.equal(out, want)
    assert torch.equal(y, hd.fmmoe_moe_forward(desc, ws, x, mask, B.FLAG_REDUCE_ON | B.FLAG_RESIDUAL))


@pytest.mark.parametrize("T,E,K,Ns,fp8", [(16, 8, 6, 2, False), (16, 8, 7, 2, False), (17, 8, 5, 1, False), (12, 4, 2, 0, False),
                                          (16, 8, 6, 1, True), (16, 16, 8, 1, True), (17, 8, 2, 0, True)])
def test_few_tokens_have_a_ring_of_their_own(T, E, K, Ns, fp8):
    """Up to 16 tokens with up to 96 pairs: more and smaller stages.  Both sides, experts that take all sixteen rows, odd numbers of k-blocks."""
    H, I_, Is = 384, 384 if fp8 else 320, 128 if fp8 else 192
    r = np.random.default_rng(T + E + K)
    w = random_layer(r, "bf16", H, E, I_, Ns, Is)
    w["router_b"] = np.where(np.arange(E) < 2, 20.0, 0.0).astype(np.float32)      # every token takes the first two
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    mask = (r.random(T) < 0.5).astype(np.uint8)
    if fp8:
        w, packed = I.weights_to_fp8(w)
        wd = upload_weights_fp8(w, packed, "bf16", "cuda")
    else:
        wd = upload_weights(w, "bf16")
    desc = B.make_desc(H, E, I_, Ns, Is if Ns else 0, K, 2, torch.bfloat16, B.WEIGHTS_FP8_BLOCK128 if fp8 else B.WEIGHTS_AS_DTYPE)
    hd = handle()
    ws = B.make_weights(wd)
    for flags in (B.FLAG_REDUCE_ON | B.FLAG_RESIDUAL, B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC):
        route = {"logits": torch.empty(T, E, dtype=torch.float32, device="cuda")}
        out = hd.fmmoe_moe_forward(desc, ws, dev(x, torch.bfloat16), dev(mask), flags, route=route)
        hd.check_status()
        ref = O.moe_forward(x, mask, w, K, 2, True, add_residual=bool(flags & B.FLAG_RESIDUAL), logits32=host(route["logits"]))
        assert row_rel_err(host(out), ref["out"]) < 2e-2


def test_layer_is_not_disturbed_by_a_status_nobody_has_read():
    """A pruning call whose mask contradicts its count leaves a status; the layers behind it, whose GEMM-2 waits for GEMM-1's rows, run as ever."""
    r = np.random.default_rng(171)
    H, E, I_, K = 2048, 16, 256, 6
    hd = B.Handle(0)
    ws = B.make_weights(upload_weights(random_layer(r, "bf16", H, E, I_, 2, 128), "bf16"))
    desc = B.make_desc(H, E, I_, 2, 128, K, 3, torch.bfloat16)
    xs = [dev(I.round_to_storage(r.standard_normal((T, H)), "bf16"), torch.bfloat16) for T in (1, 3, 200)]
    masks = [dev((r.random(x.shape[0]) < 0.5).astype(np.uint8)) for x in xs]
    want = [hd.fmmoe_moe_forward(desc, ws, x, m, B.FLAG_REDUCE_ON) for x, m in zip(xs, masks)]
    hd.check_status()
    probs = torch.softmax(torch.randn(90, E, device="cuda"), dim=1)
    hd.fmmoe_prune_visual(B.prune_params(3, 0.1), probs, None, torch.zeros(90, 64, dtype=torch.bfloat16, device="cuda"),
                          torch.zeros(90, dtype=torch.uint8, device="cuda"), [0, 90], [60], [30])      # no vision token where 60 are named
    for _ in range(5):
        assert all(torch.equal(w, hd.fmmoe_moe_forward(desc, ws, x, m, B.FLAG_REDUCE_ON)) for w, x, m in zip(want, xs, masks))
    assert hd.get_status() == 6 and hd.get_status() == 0
    hd.close()


@pytest.mark.parametrize("T,H,E,K,I_,Ns", [
    (5, 64, 8, 2, 1300, 0), (256, 256, 8, 2, 512, 0), (40, 132, 4, 1, 260, 0), (300, 260, 6, 3, 500, 1), (24, 128, 8, 4, 512, 2)])
def test_deterministic_fp32_layers_repeat_bit_for_bit(T, H, E, K, I_, Ns):
    """At shapes where GEMM-2 of the default combine shares the contraction out over CTAs whose sums are added in any order (two or more slabs
    of 128, tiles that leave SMs idle): with FLAG_DETERMINISTIC nothing depends on an order."""
    r = np.random.default_rng(T + I_)
    w = random_layer(r, "f32", H, E, I_, Ns, 256)
    x = r.standard_normal((T, H)).astype(np.float32)
    mask = (r.random(T) < 0.5).astype(np.uint8)
    desc = B.make_desc(H, E, I_, Ns, 256 if Ns else 0, K, 1, torch.float32)
    ws, xd, md = B.make_weights(upload_weights(w, "f32")), dev(x), dev(mask)
    for flags in (B.FLAG_REDUCE_ON | B.FLAG_DETERMINISTIC, B.FLAG_REDUCE_ON | B.FLAG_RESIDUAL | B.FLAG_DETERMINISTIC):
        want = handle().fmmoe_moe_forward(desc, ws, xd, md, flags)
        handle().check_status()
        assert row_rel_err(host(want), O.moe_forward(x, mask, w, K, 1, True, add_residual=bool(flags & B.FLAG_RESIDUAL))["out"]) < 1e-4
        for _ in range(40):
            assert torch.equal(want, handle().fmmoe_moe_forward(desc, ws, xd, md, flags))

"""GPU parity: routing-aware pruning (Eq. 6-18 + drop rule) through the C ABI against the
CPU oracle.  Keep-sets, kinds and offsets are compared bit-exactly (both sides rank
fp64-accumulated scores rounded once to fp32); rows within 2e-2 (bf16) / 1e-4 (fp32)."""
import numpy as np
import pytest
import torch

from oracle import fmmoe_oracle as O
from paper_2511_17885_b200 import binding as B
from paper_2511_17885_b200 import inputs as I
from gpu_util import dev, handle, host, row_rel_err, TDT

pytestmark = pytest.mark.gpu


def softmax_rows(r, n, e, smooth=None):
    z = r.standard_normal((n, e)).astype(np.float32)
    if smooth is not None:
        z = smooth
    z = z - z.max(1, keepdims=True)
    p = np.exp(z)
    return (p / p.sum(1, keepdims=True)).astype(np.float32)


def check_prune(dtype, seq_lens, H, E, W, retain, gamma, alpha, use_attn, sim_mode=0, merge_mode=0, seed=0,
                masks=None, contiguous_vision=False):
    r = np.random.default_rng(seed)
    T = int(sum(seq_lens))
    seq_off = np.concatenate([[0], np.cumsum(seq_lens)]).astype(np.int64)
    if masks is None:
        if contiguous_vision:
            mask = np.concatenate([(np.arange(L) < int(L * 0.9)).astype(np.uint8) for L in seq_lens])
        else:
            mask = I.interleaved_mask(T, r)
    else:
        mask = masks
    x = I.round_to_storage(r.standard_normal((T, H)) * (1 + r.random((T, 1))), dtype)
    # smooth logits so that neighbouring rows are similar, like vision tokens
    base = np.cumsum(0.3 * r.standard_normal((T, E)), axis=0).astype(np.float32)
    probs = softmax_rows(r, T, E, smooth=base)
    attn = r.random(T).astype(np.float32) if use_attn else None
    n_vis = np.array([int(mask[seq_off[b]:seq_off[b + 1]].sum()) for b in range(len(seq_lens))], np.int64)
    n_ret = I.retain_counts(n_vis, retain)
    p = B.prune_params(W, gamma, alpha, sim_mode, merge_mode)
    out = handle().fmmoe_prune_visual(p, dev(probs), dev(attn), dev(x, TDT[dtype]), dev(mask), seq_off, n_vis, n_ret)
    handle().check_status()
    ref = O.prune_visual(x, mask, probs, attn, seq_off, n_ret, W, alpha, gamma, sim_mode, merge_mode)
    assert out["out_seq_off"] == ref["out_seq_off"].tolist()
    assert np.array_equal(host(out["keep_idx"]), ref["keep_idx"])          # bit-exact keep-set
    assert np.array_equal(host(out["kind"]), ref["kind"])
    assert np.array_equal(host(out["is_visual_out"]), ref["is_visual_out"])
    y = host(out["x_out"])
    kept = ref["kind"] != 2
    assert np.array_equal(y[kept], x[ref["keep_idx"][kept]])                # copied rows are exact
    tol = 2e-2 if dtype == "bf16" else 1e-4
    assert row_rel_err(y, ref["x_out"]) < tol
    for b in range(len(seq_lens)):
        kc, m, d = B.fmmoe_prune_kept_count(int(n_vis[b]), int(n_ret[b]), p)
        assert (m, d, kc) == O.prune_counts(int(n_vis[b]), int(n_ret[b]), W, gamma, merge_mode)
    return out, ref


@pytest.mark.parametrize("W", [2, 3, 5, 8])
@pytest.mark.parametrize("use_attn", [False, True])
def test_prune_small(W, use_attn):
    check_prune("bf16", [301, 77, 512], 128, 24, W, 0.5, 0.08, 0.6, use_attn, seed=W)


@pytest.mark.parametrize("sim_mode,merge_mode", [(1, 0), (0, 1), (0, 2), (1, 2)])
def test_prune_modes(sim_mode, merge_mode):
    check_prune("bf16", [400, 333], 64, 40, 5, 0.4, 0.1, 0.5, True, sim_mode, merge_mode, seed=11)
    check_prune("f32", [260], 32, 9, 3, 0.25, 0.2, 0.7, False, sim_mode, merge_mode, seed=12)


def test_prune_identity_and_degenerate():
    out, ref = check_prune("bf16", [200, 100], 64, 16, 5, 1.0, 0.05, 0.5, True, seed=20)     # 100% retention
    assert out["x_out"].shape[0] == 300
    check_prune("bf16", [200], 64, 16, 5, 0.99, 0.05, 0.5, True, seed=21)                  # eps <= W: identity
    check_prune("bf16", [64], 64, 16, 5, 0.5, 0.0, 1.0, False, seed=22, masks=np.zeros(64, np.uint8))   # no vision
    check_prune("bf16", [7, 3], 64, 16, 5, 0.5, 0.05, 1.0, False, seed=23, masks=np.ones(10, np.uint8))  # tiny
    check_prune("bf16", [300], 64, 16, 4, 0.02, 0.9, 1.0, False, seed=24, masks=np.ones(300, np.uint8))  # gamma clamped
    check_prune("bf16", [300], 64, 16, 4, 0.0, 0.0, 1.0, True, seed=25, masks=np.ones(300, np.uint8))    # retain 0


def test_prune_ties_go_to_lower_window():
    # identical probability rows everywhere: all S equal (=1) -> merges and drops take the lowest windows
    T, H, E, W = 120, 64, 8, 3
    r = np.random.default_rng(30)
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    probs = np.tile(softmax_rows(r, 1, E), (T, 1))
    mask = np.ones(T, np.uint8)
    p = B.prune_params(W, 0.1, 1.0)
    out = handle().fmmoe_prune_visual(p, dev(probs), None, dev(x, torch.bfloat16), dev(mask), [0, T], [T], [60])
    ref = O.prune_visual(x, mask, probs, None, [0, T], [60], W, 1.0, 0.1)
    assert np.array_equal(host(out["keep_idx"]), ref["keep_idx"])
    act = ref["per_seq"][0]["action"]
    m, d, _ = O.prune_counts(T, 60, W, 0.1)
    assert act[:m].tolist() == [1] * m and act[m:m + d].tolist() == [2] * d


@pytest.mark.parametrize("W,n_win,use_attn,sim_mode", [
    (3, 1, True, 0), (2, 1024, True, 1), (3, 1024, False, 0), (3, 1025, True, 0), (5, 1100, False, 1), (7, 700, True, 0),
    (8, 1500, True, 0), (6, 513, True, 1), (4, 33, False, 0)])
def test_selection_on_both_sides_of_a_key_per_thread_with_many_ties(W, n_win, use_attn, sim_mode):
    """Selection with one key per thread (up to 1,024 windows) and with keys in shared memory, scores from a few
    distinct values only, so that the merge and the drop bound both fall among equal scores: the keep-set must be the
    oracle's (lower window first).  Text before, between and after the vision tokens; mask counts past 4,096 tokens."""
    r = np.random.default_rng(W * 1000 + n_win)
    n_vis = n_win * W + W - 1
    mask = np.ones(n_vis + 90, np.uint8)
    mask[r.permutation(mask.size)[:90]] = 0
    T, H, E = mask.size, 64, 40
    kinds = softmax_rows(r, 4, E)                          # four routing rows; windows are drawn from few patterns
    rows = kinds[r.integers(0, 4, (6, W))][r.integers(0, 6, n_win)].reshape(n_win * W, E)
    probs = softmax_rows(r, T, E)
    vis = np.nonzero(mask)[0]
    probs[vis[:n_win * W]] = rows
    attn = np.zeros(T, np.float32)
    attn[vis] = np.repeat(r.integers(0, 5, n_win + 1), W)[:vis.size].astype(np.float32) / 64
    x = I.round_to_storage(r.standard_normal((T, H)), "bf16")
    eta = int(n_vis * 0.45)
    p = B.prune_params(W, 0.2, 0.6, sim_mode)
    out = handle().fmmoe_prune_visual(p, dev(probs), dev(attn) if use_attn else None, dev(x, torch.bfloat16), dev(mask),
                                      [0, T], [n_vis], [eta])
    handle().check_status()
    ref = O.prune_visual(x, mask, probs, attn if use_attn else None, [0, T], [eta], W, 0.6, 0.2, sim_mode)
    assert np.array_equal(host(out["keep_idx"]), ref["keep_idx"]) and np.array_equal(host(out["kind"]), ref["kind"])
    assert row_rel_err(host(out["x_out"]), ref["x_out"]) < 2e-2


def test_longest_sequence_selection_takes():
    """16,384 windows fill the shared memory that selection asks for; one more is refused."""
    W, n = 2, 2 * 16384 + 1
    check_prune("bf16", [n, 40], 8, 4, W, 0.5, 0.1, 0.6, True, seed=5, masks=np.ones(n + 40, np.uint8))
    with pytest.raises(B.FmmoeError) as e:
        check_prune("bf16", [n + 1], 8, 4, W, 0.5, 0.1, 0.6, True, seed=5, masks=np.ones(n + 1, np.uint8))
    assert e.value.status == 2


@pytest.mark.parametrize("static", [False, True])
@pytest.mark.parametrize("lens,over", [([20000], "is_visual_out"), ([3, 9000, 700, 8300], "is_visual_out"),
                                       ([90] * 70, "is_visual_out"), ([500, 400], "kind"), ([30, 12000], "shifted")])
def test_mask_compacted_in_place(lens, over, static):
    """is_visual_out (or kind, or a mask that starts inside the other) over is_visual: selection reads the mask of a run of
    more than eight tokens a second time, and a sequence's output lies over the mask of the one before, so nothing may be
    written there before every sequence of the launch has been selected."""
    r = np.random.default_rng(sum(lens))
    T, H, E, W = sum(lens), 64, 16, 3
    seq_off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    mask = (r.random(T) < 0.85).astype(np.uint8)
    n_vis = [int(mask[seq_off[b]:seq_off[b + 1]].sum()) for b in range(len(lens))]
    n_ret = [v // 3 for v in n_vis]
    x = dev(I.round_to_storage(r.standard_normal((T, H)), "bf16"), torch.bfloat16)
    probs, attn = dev(softmax_rows(r, T, E)), dev(r.random(T).astype(np.float32))
    p = B.prune_params(W, 0.1, 0.6)
    h = handle()
    ref = h.fmmoe_prune_visual(p, probs, attn, x, dev(mask), seq_off, n_vis, n_ret)
    _, so, nv, nr, oo, t_out = B._prune_layout(p, seq_off, n_vis, n_ret)
    buf = torch.zeros(T + 64, dtype=torch.uint8, device="cuda")
    m = buf[:T]
    m.copy_(dev(mask))
    vis_out = torch.empty(t_out, dtype=torch.uint8, device="cuda")
    kind = torch.empty_like(vis_out)
    if over == "is_visual_out":
        vis_out = m[:t_out]
    elif over == "kind":
        kind = m[:t_out]
    else:
        vis_out = buf[64:64 + t_out]
    keep_idx = torch.empty(t_out, dtype=torch.int32, device="cuda")
    x_out = torch.empty((t_out, H), dtype=torch.bfloat16, device="cuda")
    args = (h._h, p, B._ptr(probs), E, B._ptr(attn), B._ptr(x), 1, H, B._ptr(m), so, nv, nr, len(lens), B._ptr(x_out),
            B._ptr(vis_out), B._ptr(keep_idx), B._ptr(kind), oo)
    if static:
        st = B.lib().fmmoe_prune_visual_static(*args, B._stream())
    else:
        wsp, wsn = h._ws_args(int(B.lib().fmmoe_prune_workspace_bytes(T, len(lens))))
        st = B.lib().fmmoe_prune_visual(*args, wsp, wsn, B._stream())
    assert st == 0
    h.check_status()
    assert list(oo) == ref["out_seq_off"]
    assert torch.equal(vis_out, ref["is_visual_out"]) and torch.equal(kind, ref["kind"])
    assert torch.equal(keep_idx, ref["keep_idx"]) and torch.equal(x_out, ref["x_out"])


@pytest.mark.parametrize("H,dtype", [(2056, "bf16"), (1028, "f32"), (8, "bf16")])
def test_merged_rows_longer_than_a_cta_keeps_in_registers(H, dtype):
    check_prune(dtype, [401, 77], H, 24, 5, 0.5, 0.2, 0.7, True, seed=H)


def test_prune_many_sequences_over_launch_chunks():
    lens = [50 + (i % 7) * 9 for i in range(70)]          # more than 64 sequences
    check_prune("bf16", lens, 64, 12, 3, 0.5, 0.05, 0.9, True, seed=40)


def test_prune_c0_and_c3_keep_sets():
    """Keep-sets on the routing probabilities the GPU router itself produces (C0 fp32, C3 sweep)."""
    from gpu_util import upload_weights, desc_of
    for cfg in (I.C0, I.C3):
        x, m, seq_off, n_vis = I.make_tokens(cfg)
        w = I.make_weights(cfg)
        wd = upload_weights(w, cfg.dtype); ws = B.make_weights(wd)
        xd, md = dev(x, TDT[cfg.dtype]), dev(m)
        rt = handle().fmmoe_route(desc_of(cfg), ws, xd, md, B.FLAG_REDUCE_ON, want=("probs", "topk_idx", "topk_w"))
        probs = host(rt["probs"])
        attn = I.make_attention_importance(cfg)
        for pc in cfg.prune:
            n_ret = I.retain_counts(n_vis, pc.retain)
            for a in (None, attn):
                p = B.prune_params(pc.window, pc.gamma, pc.alpha)
                out = handle().fmmoe_prune_visual(p, rt["probs"], dev(a), xd, md, seq_off, n_vis, n_ret)
                handle().check_status()
                ref = O.prune_visual(x, m, probs, a, seq_off, n_ret, pc.window, pc.alpha, pc.gamma)
                assert np.array_equal(host(out["keep_idx"]), ref["keep_idx"])
                assert np.array_equal(host(out["kind"]), ref["kind"])
                assert row_rel_err(host(out["x_out"]), ref["x_out"]) < (2e-2 if cfg.dtype == "bf16" else 1e-4)
    # kept counts of the sweep
    p = B.prune_params(5, 0.025)
    assert B.fmmoe_prune_kept_count(3328, 2496, p)[0] == 2500
    assert B.fmmoe_prune_kept_count(3328, 1664, B.prune_params(5, 0.05))[0] == 1666
    assert B.fmmoe_prune_kept_count(3328, 832, B.prune_params(5, 0.1))[0] == 836


@pytest.mark.parametrize("static", [False, True])
def test_mask_one_bit_short_of_n_vis_is_reported_not_followed(static):
    """The host says a sequence holds n_vis vision tokens, the mask sets one byte fewer.  The pass must end with
    FMMOE_ERR_INTERNAL from the status word - and must not index probs or x with list entries it never wrote,
    whatever the scratch held before (here: the leftovers of a larger earlier call, or a poisoned workspace).
    The next ordinary call on the same handle is unaffected."""
    h = handle()
    r = np.random.default_rng(77)
    H, E, W = 128, 16, 3
    p = B.prune_params(W, 0.1)
    # an earlier, longer call leaves large token indices behind in the shared scratch
    check_prune("bf16", [3000], H, E, W, 0.5, 0.1, 1.0, False, seed=78)
    L = 400
    mask = np.zeros(L, np.uint8); mask[:301] = 1
    n_vis_true = 301
    x = dev(I.round_to_storage(r.standard_normal((L, H)), "bf16"), torch.bfloat16)
    probs = dev(softmax_rows(r, L, E))
    bad = mask.copy(); bad[300] = 0                         # one set byte fewer than the count the host passes
    kept, _, _ = B.fmmoe_prune_kept_count(n_vis_true, 150, p)
    t_out = L - n_vis_true + kept
    if static:
        x_out = torch.zeros((t_out, H), dtype=torch.bfloat16, device="cuda")
        h.fmmoe_prune_visual_static(p, probs, None, x, dev(bad), [0, L], [n_vis_true], [150], x_out)
    else:
        h._ws = None                                        # a fresh workspace, poisoned with out-of-range indices
        ws = h.workspace(int(B.lib().fmmoe_prune_workspace_bytes(L, 1)))
        ws.fill_(0x7f)                                      # every int32 word reads 0x7f7f7f7f
        out = h.fmmoe_prune_visual(p, probs, None, x, dev(bad), [0, L], [n_vis_true], [150])
        assert out["x_out"].shape[0] == t_out
    assert h.get_status() == 6                              # FMMOE_ERR_INTERNAL, read and cleared
    torch.cuda.synchronize()                                # no fault: the context is still usable
    # the consistent call right after it passes parity
    check_prune("bf16", [L], H, E, W, 0.5, 0.1, 1.0, False, seed=79)


@pytest.mark.parametrize("lens,W,use_attn", [
    ([1024], 8, True), ([1025], 8, True),                        # tokens a small selection CTA takes
    ([514, 40], 2, True), ([520, 40], 2, False),                 # 256 and 260 windows
    ([1, 0, 300], 3, True), ([700] * 3, 5, False)])
def test_selection_on_both_sides_of_a_small_cta(lens, W, use_attn):
    """Up to 1,024 tokens and 256 windows a sequence selection runs in CTAs of 256 threads, else of 1,024."""
    T = sum(lens)
    mask = np.ones(T, np.uint8)
    if lens[0] == 514:
        mask[512:514] = 0
    check_prune("bf16", lens, 64, 16, W, 0.4, 0.1, 0.6, use_attn, seed=T + W, masks=mask)


@pytest.mark.parametrize("lens", [[8192, 5], [8193], [1024 * 9 + 1, 9000]])
def test_selection_on_both_sides_of_eight_tokens_a_thread(lens):
    """Up to eight tokens a thread stay in registers, the others are read again: ragged masks over runs of 8, 9 and 10."""
    T = sum(lens)
    mask = (np.arange(T) % 7 != 3).astype(np.uint8)
    check_prune("bf16", lens, 8, 16, 3, 0.4, 0.1, 0.6, True, seed=T, masks=mask)


def test_selection_sees_the_mask_of_its_own_call():
    """Calls back to back on the same buffers, masks and probabilities overwritten on the stream in front of every one: each works on its own, whose
    scores and selection start while the call before may still run."""
    r = np.random.default_rng(77)
    T, H, E, W = 900, 64, 16, 3
    p = B.prune_params(W, 0.1, 0.6)
    x = dev(I.round_to_storage(r.standard_normal((T, H)), "bf16"), torch.bfloat16)
    staged = []
    for i in range(4):
        probs = softmax_rows(r, T, E, smooth=np.cumsum(0.3 * r.standard_normal((T, E)), axis=0).astype(np.float32))
        mask = (r.random(T) < (0.9 - 0.2 * i)).astype(np.uint8)
        staged.append((dev(probs), dev(mask), [int(mask.sum())], [int(mask.sum()) // 2]))
    h = handle()
    want = [h.fmmoe_prune_visual(p, pr, None, x, m, [0, T], nv, nr) for pr, m, nv, nr in staged]
    pb, mb, got = torch.empty_like(staged[0][0]), torch.empty_like(staged[0][1]), []
    for pr, m, nv, nr in staged:
        pb.copy_(pr); mb.copy_(m)
        got.append(h.fmmoe_prune_visual(p, pb, None, x, mb, [0, T], nv, nr))
    h.check_status()
    for a, b in zip(want, got):
        for k in ("x_out", "keep_idx", "kind", "is_visual_out"):
            assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("lens,texts,W", [
    ([40], [24], 3), ([2], [62], 5), ([1500], [100], 3), ([1500], [100], 8), ([300] * 6, [5] * 6, 5), ([5000], [60], 8)])
def test_layer_with_its_stage_is_the_layer_and_the_stage(lens, texts, W):
    """Beside a pruning stage the small-M expert GEMMs run on fewer SMs, by the number of windows: one to six fewer here, with routed and
    shared tiles in the first round.  Rows and pruned rows are bit for bit those of the two calls one after the other."""
    r = np.random.default_rng(sum(lens) + W)
    off = np.concatenate([[0], np.cumsum(np.array(lens) + np.array(texts))]).tolist()
    T, H, E, I_, K = off[-1], 128, 160, 64, 2
    w = {"router_w": r.standard_normal((E, H)) * 0.1, "router_b": None, "w_gate": r.standard_normal((E, I_, H)) * 0.1, "w_up": r.standard_normal((E, I_, H)) * 0.1,
         "w_down": r.standard_normal((E, H, I_)) * 0.1, "ws_gate": r.standard_normal((1, 128, H)) * 0.1, "ws_up": r.standard_normal((1, 128, H)) * 0.1,
         "ws_down": r.standard_normal((1, H, 128)) * 0.1}
    wd = {k: v if v is None else dev(v.astype(np.float32), torch.bfloat16) for k, v in w.items()}
    desc, ws = B.make_desc(H, E, I_, 1, 128, K, 1, torch.bfloat16), B.make_weights(wd)
    x = dev(r.standard_normal((T, H)).astype(np.float32), torch.bfloat16)
    mask = dev(np.concatenate([np.concatenate([np.ones(v, np.uint8), np.zeros(t, np.uint8)]) for v, t in zip(lens, texts)]))
    p, nr = B.prune_params(W, 0.1, 0.6), [v // 2 for v in lens]
    h = B.Handle(0)
    route = {"probs": torch.empty(T, E, dtype=torch.float32, device="cuda")}
    want = h.fmmoe_moe_forward(desc, ws, x, mask, B.FLAG_REDUCE_ON, route=route)
    rows = h.fmmoe_prune_visual(p, route["probs"], None, want, mask, off, lens, nr)
    for _ in range(3):
        out, route2 = torch.empty_like(x), {"probs": torch.empty(T, E, dtype=torch.float32, device="cuda")}
        got = h.fmmoe_moe_forward_prune(desc, ws, x, mask, B.FLAG_REDUCE_ON, out, route2, p, None, off, lens, nr)
        h.check_status()
        assert torch.equal(out, want)
        for k in ("x_out", "keep_idx", "kind", "is_visual_out"):
            assert torch.equal(got[k], rows[k]), k
    h.close()


@pytest.mark.parametrize("W,lens", [(5, [11840]), (5, [11841, 30]), (8, [9472]), (8, [9473]), (8, [40, 41]), (4, [500]), (6, [700])])
def test_window_scores_with_few_and_with_many_ctas(W, lens):
    """A stage alone scores W = 5 and 8 in CTAs of more registers up to 296 and 148 of them (a full chip): both sides, eight windows a CTA."""
    check_prune("bf16", lens, 16, 24, W, 0.5, 0.05, 0.6, True, seed=sum(lens) + W)

"""GPU parity: router + top-k + gates (Eq. 1-3, 5) and the permutation, through the C ABI,
against the CPU oracle on the same seeded inputs.  Selections and permutation indices are
compared bit-exactly (the oracle takes its decision on the kernel's own fp32 logits);
floating-point outputs within tolerances stated per test."""
import numpy as np
import pytest
import torch

from oracle import fmmoe_oracle as O
from paper_2511_17885_b200 import binding as B
from paper_2511_17885_b200 import inputs as I
from gpu_util import dev, handle, host, TDT

pytestmark = pytest.mark.gpu

CASES = [
    # dtype, T, H, E, K, Kv, bias, reduce_on
    ("f32", 256, 256, 8, 2, 1, False, 1),
    ("f32", 77, 100, 5, 3, 2, True, 1),
    ("bf16", 2432, 2048, 64, 6, 3, True, 1),
    ("bf16", 1000, 512, 72, 6, 2, False, 1),
    ("bf16", 333, 256, 128, 8, 4, False, 1),
    ("bf16", 65, 128, 200, 16, 1, True, 1),
    ("bf16", 31, 64, 256, 8, 8, False, 0),
    ("bf16", 1, 64, 33, 4, 0, False, 1),
]


def check_route(dtype, T, H, E, K, Kv, bias, reduce_on, seed=0, mask=None, x=None, w=None, b=None, launches=None):
    r = np.random.default_rng(seed)
    x = I.round_to_storage(r.standard_normal((T, H)), dtype) if x is None else x
    w = I.round_to_storage(0.05 * r.standard_normal((E, H)), dtype) if w is None else w
    b = (0.5 * r.standard_normal(E)).astype(np.float32) if (bias and b is None) else b
    mask = (r.random(T) < 0.7).astype(np.uint8) if mask is None else mask
    td = TDT[dtype]
    desc = B.make_desc(H, E, 64, 1 if Kv == 0 else 0, 64, K, Kv, td)
    wd = {"router_w": dev(w, td), "router_b": dev(b)}
    ws = B.make_weights(wd)
    before = handle().launch_count()
    out = handle().fmmoe_route(desc, ws, dev(x, td), dev(mask), B.FLAG_REDUCE_ON if reduce_on else 0)
    handle().check_status()
    assert launches is None or handle().launch_count() - before == launches
    g = {k: host(v) for k, v in out.items()}
    ref = O.route(x, w, b, mask, K, Kv, bool(reduce_on), logits32=g["logits"])
    # logits: fp32 accumulation of exact products vs fp64
    scale = np.abs(ref["logits"]).max() + 1e-30
    assert np.abs(g["logits"] - ref["logits"]).max() / scale < 2e-5
    assert np.abs(g["probs"] - ref["probs"]).max() < 2e-5
    assert np.array_equal(g["topk_idx"], ref["topk_idx"])                       # bit-exact selection
    assert np.abs(g["topk_w"] - ref["topk_w"]).max() < 2e-5
    # independent selection check on the oracle's own logits: any disagreement must be a near-tie
    ind = O.route(x, w, b, mask, K, Kv, bool(reduce_on))
    bad = np.nonzero((ind["topk_idx"] != g["topk_idx"]).any(axis=1))[0]
    for t in bad:
        z = np.sort(ref["logits"][t])[::-1]
        k_t = int(ref["k_t"][t])
        gaps = np.abs(np.diff(z[:k_t + 1]))
        assert gaps.min() < 1e-4 * scale, f"token {t}: selection differs without a near-tie"
    assert len(bad) <= max(1, T // 100)
    # permutation: bit-exact
    off, row_token, inv = O.permutation(ref["topk_idx"], E)
    assert np.array_equal(g["expert_off"], off)
    P = off[-1]
    assert np.array_equal(g["row_token"][:P], row_token)
    assert np.array_equal(g["inv_row"], inv)
    return g, ref


@pytest.mark.parametrize("case", CASES)
def test_route_parity(case):
    check_route(*case)


@pytest.mark.parametrize("T,H,E,K,Kv", [
    (32, 256, 64, 6, 3), (33, 256, 8, 2, 1), (128, 512, 128, 8, 4), (129, 256, 128, 8, 4), (256, 256, 255, 16, 5),
    (257, 256, 64, 6, 3),                                        # contraction split over four CTAs: fused up to 256 tokens
    (500, 128, 192, 16, 7), (512, 384, 40, 4, 4), (513, 128, 40, 4, 2),        # over two: up to 512
    (1000, 64, 192, 16, 3), (1024, 192, 256, 5, 2), (1025, 64, 33, 3, 1)])     # not split: up to 1,024
def test_permutation_inside_the_router_up_to_a_cluster_of_eight(T, H, E, K, Kv):
    """Both sides of the sizes up to which the router's own cluster writes the permutation (one launch; beyond, a second
    one), for each split of the contraction, with the largest shared-memory demand (192 experts, top-16): same stable
    grouping, bit for bit."""
    check_route("bf16", T, H, E, K, Kv, True, 1, seed=T + E, launches=2 if T in (257, 513, 1025) else 1)


@pytest.mark.parametrize("dtype,T,one_expert", [
    ("bf16", 32768, True), ("bf16", 32768, False), ("bf16", 32769, True), ("bf16", 32769, False), ("bf16", 40000, False),
    ("f32", 8192, False), ("f32", 8193, True), ("f32", 8193, False)])
def test_permutation_on_both_sides_of_256_token_blocks(dtype, T, one_expert):
    """Up to 256 token blocks (of 128 tokens, fp32: 32) one kernel sums the count table as pairs of 16-bit halves, fullest
    when every token takes one expert; beyond, a scan and a scatter kernel."""
    b = np.zeros(8, np.float32)
    b[5] = 8.0 if one_expert else 0.0          # the other logits have a standard deviation of 0.4
    g, _ = check_route(dtype, T, 64, 8, 2, 1, True, 1, seed=T, b=b, launches=2 if T in (8192, 32768) else 3)
    assert not one_expert or g["expert_off"][6] - g["expert_off"][5] == T


def test_route_exact_ties_go_to_lower_index():
    # duplicate router rows => exactly equal logits
    r = np.random.default_rng(5)
    T, H, E = 64, 128, 16
    w = I.round_to_storage(0.05 * r.standard_normal((E, H)), "bf16")
    w[9] = w[2]; w[11] = w[2]; w[5] = w[4]
    g, ref = check_route("bf16", T, H, E, 4, 2, False, 1, w=w)
    z = g["logits"]
    assert np.array_equal(z[:, 9], z[:, 2]) and np.array_equal(z[:, 11], z[:, 2])
    for t in range(T):
        sel = g["topk_idx"][t][g["topk_idx"][t] >= 0].tolist()
        if 9 in sel:
            assert 2 in sel and sel.index(2) < sel.index(9)
        if 11 in sel:
            assert 9 in sel and sel.index(9) < sel.index(11)


def test_route_all_visual_all_text_and_constant_logits():
    check_route("bf16", 100, 64, 32, 4, 2, False, 1, mask=np.ones(100, np.uint8))
    check_route("bf16", 100, 64, 32, 4, 2, False, 1, mask=np.zeros(100, np.uint8))
    # zero router => all logits equal => experts 0..k-1, uniform gates
    g, _ = check_route("f32", 40, 64, 10, 3, 2, False, 1, w=np.zeros((10, 64), np.float32))
    assert (g["topk_idx"][:, 0] == 0).all() and (g["topk_idx"][:, 1] == 1).all()


def test_route_config_sequences():
    for cfg in (I.C0, I.C2):
        x, m, _, _ = I.make_tokens(cfg)
        w = I.make_weights(cfg)
        check_route(cfg.dtype, cfg.n_tokens, cfg.hidden, cfg.n_experts, cfg.top_k, cfg.top_k_vis, False, 1,
                    mask=m, x=x, w=w["router_w"], b=w["router_b"])


def test_route_empty_and_invalid():
    h = handle()
    desc = B.make_desc(64, 8, 64, 0, 0, 2, 1, torch.bfloat16)
    w = B.make_weights({"router_w": torch.zeros(8, 64, dtype=torch.bfloat16, device="cuda")})
    out = h.fmmoe_route(desc, w, torch.zeros(0, 64, dtype=torch.bfloat16, device="cuda"),
                        torch.zeros(0, dtype=torch.uint8, device="cuda"), 1)
    assert out["topk_idx"].shape == (0, 2)
    bad = B.make_desc(64, 8, 64, 0, 0, 2, 3, torch.bfloat16)       # K_v > K
    with pytest.raises(B.FmmoeError) as e:
        h.fmmoe_route(bad, w, torch.zeros(4, 64, dtype=torch.bfloat16, device="cuda"),
                      torch.zeros(4, dtype=torch.uint8, device="cuda"), 1)
    assert e.value.status == 1
    bad2 = B.make_desc(64, 8, 64, 0, 0, 2, 0, torch.bfloat16)      # K_v = 0 without shared experts
    assert B.fmmoe_workspace_bytes(bad2, 4) == 0
    un = B.make_desc(72, 8, 64, 0, 0, 2, 1, torch.bfloat16)        # H % 64 != 0 on the bf16 path
    with pytest.raises(B.FmmoeError) as e:
        h.fmmoe_route(un, w, torch.zeros(4, 72, dtype=torch.bfloat16, device="cuda"),
                      torch.zeros(4, dtype=torch.uint8, device="cuda"), 1)
    assert e.value.status == 2


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_route_non_finite_activations_still_give_valid_distinct_experts(dtype):
    """Overflowed activations upstream (inf / nan rows) must not turn into out-of-range expert indices:
    the router clamps non-finite logits before it selects, so every token gets k distinct experts in
    [0, E) and the permutation stays consistent."""
    r = np.random.default_rng(8)
    T, H, E, K, Kv = 300, 128, 24, 4, 2
    x = I.round_to_storage(r.standard_normal((T, H)), dtype)
    x[5] = np.inf; x[17] = np.nan; x[40, ::2] = -np.inf; x[41] = 3e38
    w = I.round_to_storage(0.05 * r.standard_normal((E, H)), dtype)
    mask = (r.random(T) < 0.5).astype(np.uint8)
    td = TDT[dtype]
    desc = B.make_desc(H, E, 64, 0, 64, K, Kv, td)
    ws = B.make_weights({"router_w": dev(w, td)})
    out = handle().fmmoe_route(desc, ws, dev(x, td), dev(mask), B.FLAG_REDUCE_ON)
    handle().check_status()
    idx = host(out["topk_idx"])
    for t in range(T):
        k = Kv if mask[t] else K
        sel = idx[t, :k]
        assert (sel >= 0).all() and (sel < E).all() and len(set(sel.tolist())) == k, (t, sel)
        assert (idx[t, k:] == -1).all()
    off, row_token, inv = O.permutation(idx, E)
    assert np.array_equal(host(out["expert_off"]), off)
    assert np.array_equal(host(out["row_token"])[:off[-1]], row_token)
    assert np.array_equal(host(out["inv_row"]), inv)


@pytest.mark.parametrize("T,H,cta,k_block", [
    (200, 256, 0, 0), (200, 256, 5, 0), (700, 64, 3, 0), (700, 256, 0, 0), (1100, 64, 8, 0),
    (200, 256, 0, -1), (200, 256, 5, -1), (700, 64, 3, -1)])       # behind the counts, which its peers have by then
def test_a_router_wait_that_runs_out_leaves_a_record_that_can_be_followed(T, H, cta, k_block):
    """One router CTA gives up (its own cluster, the cluster that also permutes, or a grid without clusters).  Its tokens
    read as having selected nothing; every other index of the record is in range, also where buffers and workspace
    held large numbers before; the layer behind it runs to its end; the status is reported once; the next call is right."""
    h = B.Handle(0)
    r = np.random.default_rng(T + cta)
    E, K, Kv = 12, 4, 2
    x = dev(I.round_to_storage(r.standard_normal((T, H)), "bf16"), torch.bfloat16)
    mask = dev((r.random(T) < 0.7).astype(np.uint8))
    bf = lambda *s: dev(I.round_to_storage(0.05 * r.standard_normal(s), "bf16"), torch.bfloat16)
    ws = B.make_weights({"router_w": bf(E, H), "w_gate": bf(E, 64, H), "w_up": bf(E, 64, H), "w_down": bf(E, H, 64)})
    desc = B.make_desc(H, E, 64, 0, 0, K, Kv, torch.bfloat16)
    split = 4 if H == 256 else 1                         # H = 256: four CTAs share a tile of 128 tokens
    rows = 128 // split
    mine = np.arange(T)
    mine = (mine // 128 * split + mine % 128 // rows) == cta
    assert mine.any()
    for layer in (False, True):
        h.workspace(B.fmmoe_workspace_bytes(desc, T, 0)).fill_(0x7f)
        rec = {k: torch.full(s, 0x7f7f7f7f, dtype=torch.int32, device="cuda") for k, s in
               (("topk_idx", (T, K)), ("expert_off", (E + 1,)), ("row_token", (T * K,)), ("inv_row", (T, K)))}
        h.fmmoe_test_expire_route_wait(3_000_000, cta, k_block)
        if layer:
            h.fmmoe_moe_forward(desc, ws, x, mask, B.FLAG_REDUCE_ON, route=rec)
        else:
            ro = B.RouteOut(**{k: v.data_ptr() for k, v in rec.items()})
            wsp, wsn = h._ws_args(B.fmmoe_workspace_bytes(desc, T, 0))
            assert B.lib().fmmoe_route(h._h, desc, ws, B._ptr(x), B._ptr(mask), T, B.FLAG_REDUCE_ON, ro, wsp, wsn, B._stream()) == 0
        assert h.get_status() == 5 and h.get_status() == 0
        idx, inv, off = host(rec["topk_idx"]), host(rec["inv_row"]), host(rec["expert_off"])
        assert (idx[mine] == -1).all() and (inv[mine] == -1).all()
        assert ((idx >= -1) & (idx < E)).all() and ((inv >= -1) & (inv < T * K)).all()
        assert (np.diff(off) >= 0).all() and off[0] == 0 and off[-1] <= T * K
        row_token = host(rec["row_token"])[:off[-1]]
        assert ((row_token >= 0) & (row_token < T)).all() and not mine[row_token].any()
    out = h.fmmoe_route(desc, ws, x, mask, B.FLAG_REDUCE_ON)
    h.check_status()
    want = O.permutation(host(out["topk_idx"]), E)
    assert (host(out["topk_idx"])[:, 0] >= 0).all() and np.array_equal(host(out["inv_row"]), want[2])
    h.close()


@pytest.mark.parametrize("T,H,E,K,Kv", [
    (300, 256, 224, 4, 2), (300, 256, 225, 4, 2),      # four CTAs a tile: partial rows are pushed up to 224 experts, read beyond
    (5249, 128, 224, 4, 2), (5249, 128, 250, 4, 2),    # two CTAs a tile (room for either); a last tile of one row
    (64, 2048, 192, 8, 4), (65, 2048, 192, 8, 4),      # pushed, though the ring keeps three stages only; read, so that it has five
    (300, 2048, 160, 8, 4), (300, 2048, 161, 8, 4),    # four stages beside the pushed rows; three
    (257, 256, 8, 2, 1), (385, 256, 64, 6, 3)])        # a last tile of one row: three CTAs of it own no rows
def test_partial_rows_reach_the_cta_that_owns_them(T, H, E, K, Kv):
    """The partial logits of a tile's CTAs, by bulk copies of the rows that exist or read through the cluster."""
    check_route("bf16", T, H, E, K, Kv, True, 1, seed=T + E)


@pytest.mark.parametrize("T,H,E,K,Kv", [
    (1, 256, 13, 5, 1), (130, 256, 7, 3, 1), (255, 128, 9, 2, 1), (900, 64, 21, 5, 2),      # the cluster permutes (4, 8, 4 and 8 CTAs)
    (300, 256, 11, 3, 1), (700, 256, 225, 3, 2), (5300, 128, 19, 7, 3)])                    # clusters of four and two, counts left to the permutation
def test_cluster_barriers_behind_uneven_loops(T, H, E, K, Kv):
    """Odd numbers of experts and selections: the lanes of a warp leave the router's strided loops, which its cluster
    barriers follow, after different numbers of turns."""
    for seed in range(3):
        check_route("bf16", T, H, E, K, Kv, True, 1, seed=T + E + seed)


@pytest.mark.parametrize("T,H,E,K,launches", [
    (256, 256, 8, 2, 1), (257, 256, 8, 2, 2),                    # eight blocks of 32 tokens: the permutation inside the router; nine
    (1, 60, 5, 5, 1), (33, 300, 9, 3, 1), (64, 64, 16, 16, 1), (40, 132, 17, 4, 1),      # shares of the contraction: four, two, one
    (200, 520, 33, 6, 1), (255, 128, 250, 8, 1),                 # more slabs than are on their way at once
    (17, 192, 16, 3, 1), (49, 192, 17, 3, 1), (272, 192, 17, 3, 2), (15, 64, 96, 4, 1), (300, 320, 130, 5, 2), (250, 100, 256, 7, 1)])      # one token a warp; two
def test_fp32_router_at_the_edges_of_its_forms(T, H, E, K, launches):
    check_route("f32", T, H, E, K, max(K // 2, 1), True, 1, seed=T + E, launches=launches)


@pytest.mark.parametrize("T,E,cta", [(200, 12, 0), (200, 12, 5), (256, 40, 7), (20, 12, 0)])
def test_an_fp32_router_that_gives_up_behind_its_counts_leaves_a_record_that_can_be_followed(T, E, cta):
    """The same for the fp32 router that does the permutation: its peers have counted the pairs of the CTA that gave up, so no expert has rows."""
    h = B.Handle(0)
    r = np.random.default_rng(T + cta)
    H, K, Kv = 64, 4, 2
    x, mask = dev(r.standard_normal((T, H)).astype(np.float32)), dev((r.random(T) < 0.7).astype(np.uint8))
    f32 = lambda *s: dev((0.05 * r.standard_normal(s)).astype(np.float32))
    ws = B.make_weights({"router_w": f32(E, H), "w_gate": f32(E, 64, H), "w_up": f32(E, 64, H), "w_down": f32(E, H, 64)})
    desc = B.make_desc(H, E, 64, 0, 0, K, Kv, torch.float32)
    mine = np.arange(T) // 32 == cta
    assert mine.any()
    for layer in (False, True):
        h.workspace(B.fmmoe_workspace_bytes(desc, T, 0)).fill_(0x7f)
        rec = {k: torch.full(s, 0x7f7f7f7f, dtype=torch.int32, device="cuda") for k, s in
               (("topk_idx", (T, K)), ("expert_off", (E + 1,)), ("row_token", (T * K,)), ("inv_row", (T, K)))}
        h.fmmoe_test_expire_route_wait(3_000_000, cta, -1)
        if layer:
            out = h.fmmoe_moe_forward(desc, ws, x, mask, B.FLAG_REDUCE_ON, route=rec)
        else:
            ro = B.RouteOut(**{k: v.data_ptr() for k, v in rec.items()})
            wsp, wsn = h._ws_args(B.fmmoe_workspace_bytes(desc, T, 0))
            assert B.lib().fmmoe_route(h._h, desc, ws, B._ptr(x), B._ptr(mask), T, B.FLAG_REDUCE_ON, ro, wsp, wsn, B._stream()) == 0
        assert h.get_status() == 5 and h.get_status() == 0
        idx, inv = host(rec["topk_idx"]), host(rec["inv_row"])
        assert (idx[mine] == -1).all() and (inv[mine] == -1).all()
        assert ((idx >= -1) & (idx < E)).all() and ((inv >= -1) & (inv < T * K)).all()
        assert (host(rec["expert_off"]) == 0).all()
    assert (host(out) == 0).all()
    out = h.fmmoe_route(desc, ws, x, mask, B.FLAG_REDUCE_ON)
    h.check_status()
    want = O.permutation(host(out["topk_idx"]), E)
    assert np.array_equal(host(out["expert_off"]), want[0]) and np.array_equal(host(out["inv_row"]), want[2])
    h.close()

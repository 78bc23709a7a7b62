"""tree_verify_attn on the GPU against the fp64 oracle (max-abs 2e-2), plus the
checks that pin the mask through the whole kernel: closed forms, leak canaries,
NaN-poisoned padding, non-ancestor perturbation, state safety."""
import math

import numpy as np
import pytest
import torch

import paper_2603_08088_b200 as tv
from oracle import tree_verify_oracle as orc
from workloads import (CONFIGS, make_case, case_to_numpy, bf16_bits, random_parent_tree, topk_expansion_tree,
                       chain_tree)
from gpu_util import to_device, f32, assert_attention_close, oracle_attention_slice, oracle_visibility, ATTN_ATOL

pytestmark = pytest.mark.gpu


def gpu_attention(case, layer=0, simt=False):
    """case: device tensors.  Returns (out, lse, anc_bits, dense) for one layer; `dense` is the ORACLE's
    mask of the same trees (the CUDA mask is checked equal to it here and then dropped), so that every
    expected value below comes from the oracle alone."""
    L, B, N, Hq, d = case["q"].shape
    Hkv, Scap = case["k_cache"].shape[2], case["k_cache"].shape[3]
    dev = case["q"].device
    W = (N + 31) // 32
    bits = torch.zeros(B, N, W, dtype=torch.int32, device=dev)
    dense = torch.zeros(B, 1, N, N, dtype=torch.uint8, device=dev)
    status = torch.zeros(B, dtype=torch.int32, device=dev)
    tv.tree_build_mask(case["parent"], case["n_nodes"], N - 1, 1, bits, status, dense_mask=dense)
    out = torch.full((B, N, Hq, d), 3.0, dtype=torch.bfloat16, device=dev)
    lse = torch.full((B, Hq, N), 3.0, dtype=torch.float32, device=dev)
    scale = d ** -0.5
    if simt:
        tv.tv_debug_attn_simt(case["q"][layer], case["k_cache"][layer], case["v_cache"][layer],
                              case["k_tree"][layer], case["v_tree"][layer], case["prefix_len"],
                              case["n_nodes"], bits, scale, out, lse=lse)
    else:
        ws = torch.zeros(max(256, tv.tv_attn_workspace_bytes(B, N, Hq, Hkv, d, Scap)), dtype=torch.uint8, device=dev)
        tv.tree_verify_attn(case["q"][layer], case["k_cache"][layer], case["v_cache"][layer],
                            case["k_tree"][layer], case["v_tree"][layer], case["prefix_len"],
                            case["n_nodes"], bits, scale, out, ws, status, lse=lse)
    torch.cuda.synchronize()
    assert (status.cpu().numpy() == 0).all(), f"status {status.cpu().numpy()}"
    dense = torch.from_numpy(oracle_visibility(case["parent"], case["n_nodes"], dense_gpu=dense, bits_gpu=bits))
    return out, lse, bits, dense


def oracle_attention(case_np, dense, layer=0):
    d = case_np["q"].shape[-1]
    return orc.tree_attention(case_np["q"][layer], case_np["k_cache"][layer], case_np["v_cache"][layer],
                              case_np["k_tree"][layer], case_np["v_tree"][layer], case_np["prefix_len"],
                              case_np["n_nodes"], dense[:, 0], d ** -0.5)


SMALL = [
    # name, base config, overrides: several key tiles, ragged tails, both head dims, G in {1,2,4}
    ("tiny_full", 0, {}),
    ("d64_g2_ragged", 0, dict(B=3, S_lo=0, S_hi=300, Scap=320, N=15)),
    ("d128_g1", 1, dict(Hq=4, Hkv=4, S_lo=129, S_hi=129, Scap=256, N=60)),
    ("d128_g4_ragged", 2, dict(B=4, Hq=8, Hkv=2, S_lo=1, S_hi=700, Scap=768, N=64)),
    ("d128_g4_n128", 3, dict(B=2, Hq=8, Hkv=2, S_lo=383, S_hi=385, Scap=512, N=128)),
    ("d128_g4_n60", 4, dict(B=3, L=2, Hq=8, Hkv=2, S_lo=100, S_hi=520, Scap=640, V=0)),
]


@pytest.mark.parametrize("name,ci,over", SMALL, ids=[s[0] for s in SMALL])
@pytest.mark.parametrize("simt", [False, True], ids=["tc", "simt"])
def test_attention_parity_small(name, ci, over, simt):
    cfg = CONFIGS[ci].scaled(**over)
    case = make_case(cfg, seed=1000 * ci + 1, ragged_nodes=(cfg.B > 1), with_logits=False)
    # rows past the prefix and padded tree slots hold NaN: they must never reach an output
    S = case["prefix_len"].numpy()
    n = case["n_nodes"].numpy()
    nan = torch.tensor(float("nan"), dtype=torch.bfloat16)
    for b in range(cfg.B):
        case["k_cache"][:, b, :, S[b]:] = nan
        case["v_cache"][:, b, :, S[b]:] = nan
        case["k_tree"][:, b, n[b]:] = nan
        case["v_tree"][:, b, n[b]:] = nan
        case["q"][:, b, n[b]:] = nan
    dcase = to_device(case)
    case_np = case_to_numpy(case)
    for layer in range(cfg.L):
        out, lse, bits, dense = gpu_attention(dcase, layer, simt=simt)
        ref_out, ref_lse = oracle_attention(case_np, dense.cpu().numpy(), layer)
        assert_attention_close(out, lse, ref_out, ref_lse, name)
        got = f32(out)
        for b in range(cfg.B):                       # padded rows are exact zeros / -inf
            assert (got[b, n[b]:] == 0).all()
            assert np.isneginf(f32(lse)[b, :, n[b]:]).all()


GROUPS = [
    # (query heads per KV head, KV heads, nodes, d): group sizes that do not divide the 128-row tile leave rows of
    # every tile unused (128 // G nodes per tile), and large groups put few nodes into a tile
    (3, 2, 50, 128), (5, 1, 30, 128), (6, 2, 64, 64), (7, 4, 26, 128), (12, 1, 21, 128), (24, 1, 11, 64),
    (128, 1, 3, 128), (7, 1, 129, 128),
]


@pytest.mark.parametrize("G,Hkv,N,d", GROUPS, ids=[f"G{g}_kv{h}_N{n}_d{d}" for g, h, n, d in GROUPS])
def test_group_sizes_that_do_not_divide_the_row_tile(G, Hkv, N, d):
    cfg = CONFIGS[0].scaled(B=3, Hq=G * Hkv, Hkv=Hkv, d=d, S_lo=0, S_hi=700, Scap=1024, N=N, D=min(6, N - 1), V=0,
                            tree="uniform")
    case = make_case(cfg, seed=4200 + G, ragged_nodes=True, with_logits=False)
    dcase = to_device(case)
    case_np = case_to_numpy(case)
    n = case["n_nodes"].numpy()
    out, lse, bits, dense = gpu_attention(dcase, 0)
    ref_out, ref_lse = oracle_attention(case_np, dense.cpu().numpy(), 0)
    assert_attention_close(out, lse, ref_out, ref_lse, f"G={G}")
    got = f32(out)
    for b in range(cfg.B):
        assert (got[b, n[b]:] == 0).all()
    # all layers in one launch and the paged layout walk the same row tiles
    L = 2
    cfg2 = cfg.scaled(L=L)
    case2 = make_case(cfg2, seed=4300 + G, ragged_nodes=True, with_logits=False)
    g2 = to_device(case2)
    B, Hq = cfg.B, cfg.Hq
    bits2 = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(g2["parent"], g2["n_nodes"], N - 1, 1, bits2, st)
    ws = torch.zeros(max(256, tv.tv_attn_workspace_bytes(B, N, Hq, Hkv, d, cfg.Scap)), dtype=torch.uint8, device="cuda")
    out2 = torch.full((L, B, N, Hq, d), 3.0, dtype=torch.bfloat16, device="cuda")
    lse2 = torch.zeros(L, B, Hq, N, device="cuda")
    tv.tree_verify_attn_layers(g2["q"], g2["k_cache"], g2["v_cache"], g2["k_tree"], g2["v_tree"], g2["prefix_len"],
                               g2["n_nodes"], bits2, d ** -0.5, out2, ws, st, lse=lse2)
    torch.cuda.synchronize()
    assert (st.cpu().numpy() == 0).all()
    vis = oracle_visibility(case2["parent"], case2["n_nodes"], bits_gpu=bits2)
    cn = case_to_numpy(case2)
    for l in range(L):
        r_out, r_lse = orc.tree_attention(cn["q"][l], cn["k_cache"][l], cn["v_cache"][l], cn["k_tree"][l], cn["v_tree"][l],
                                          cn["prefix_len"], cn["n_nodes"], vis[:, 0], d ** -0.5)
        assert_attention_close(out2[l], lse2[l], r_out, r_lse, f"G={G}, layer {l}")


@pytest.mark.parametrize("B", [33, 70, 512])
def test_many_sequences_up_to_the_maximum(B):
    """The schedule table is built 32 sequences at a time and searched per work item; the library takes up to
    512 sequences.  Short ragged sequences, so that most CTAs walk many units."""
    cfg = CONFIGS[0].scaled(B=B, Hq=4, Hkv=2, d=64, S_lo=0, S_hi=300, Scap=384, N=9, D=4, V=0, tree="uniform")
    case = make_case(cfg, seed=9000 + B, ragged_nodes=True, with_logits=False)
    dcase = to_device(case)
    out, lse, bits, dense = gpu_attention(dcase, 0)
    ref_out, ref_lse = oracle_attention(case_to_numpy(case), dense.cpu().numpy(), 0)
    assert_attention_close(out, lse, ref_out, ref_lse, f"B={B}")
    if B == 512:                # one more sequence is refused, nothing is launched
        big = CONFIGS[0].scaled(B=513, Hq=4, Hkv=2, d=64, S_lo=0, S_hi=10, Scap=128, N=9, D=4, V=0, tree="uniform")
        g = to_device(make_case(big, seed=1, with_logits=False))
        ws = torch.zeros(1 << 20, dtype=torch.uint8, device="cuda")
        st = torch.zeros(513, dtype=torch.int32, device="cuda")
        o = torch.zeros(513, 9, 4, 64, dtype=torch.bfloat16, device="cuda")
        b513 = torch.zeros(513, 9, 1, dtype=torch.int32, device="cuda")
        with pytest.raises(tv.TreeVerifyError):
            tv.tree_verify_attn(g["q"][0], g["k_cache"][0], g["v_cache"][0], g["k_tree"][0], g["v_tree"][0], g["prefix_len"],
                                g["n_nodes"], b513, 0.125, o, ws, st)


@pytest.mark.parametrize("d,G", [(128, 4), (64, 1), (128, 8)])
def test_prefix_lengths_on_and_around_tile_boundaries(d, G):
    """Prefixes of 0, 127, 128, 129, 255, 256, 257 keys and one that fills the cache to its last row: the ragged
    last prefix tile has 127, 0 (it does not exist), 1 ... valid keys.  Rows behind each prefix hold NaN."""
    S = np.array([0, 127, 128, 129, 255, 256, 257, 512], dtype=np.int32)
    B, Scap, N = len(S), 512, 33
    cfg = CONFIGS[0].scaled(B=B, Hq=2 * G, Hkv=2, d=d, S_lo=0, S_hi=Scap, Scap=Scap, N=N, D=6, V=0, tree="uniform")
    case = make_case(cfg, seed=777 + d + G, ragged_nodes=True, with_logits=False)
    case["prefix_len"] = torch.from_numpy(S.copy())
    nan = torch.tensor(float("nan"), dtype=torch.bfloat16)
    for b in range(B):
        case["k_cache"][:, b, :, S[b]:] = nan
        case["v_cache"][:, b, :, S[b]:] = nan
    out, lse, bits, dense = gpu_attention(to_device(case), 0)
    ref_out, ref_lse = oracle_attention(case_to_numpy(case), dense.cpu().numpy(), 0)
    assert_attention_close(out, lse, ref_out, ref_lse, f"d={d} G={G}")


BUDGETS = [(16, 10), (32, 10), (64, 4), (64, 16), (128, 10), (200, 12), (256, 10), (256, 16)]


@pytest.mark.parametrize("N,D", BUDGETS, ids=[f"M{n}_D{d}" for n, d in BUDGETS])
def test_budget_sweep_shapes(N, D):
    """Node budgets and depth bounds of the paper's sweep (Table 2: M in 16..256, Dmax in 4..16);
    more than 128 nodes means two tree key tiles and eight mask words per row."""
    cfg = CONFIGS[2].scaled(B=3, Hq=8, Hkv=2, S_lo=100, S_hi=420, Scap=512, N=N, D=D, tree="spine", V=0)
    case = make_case(cfg, seed=7000 + N + D, ragged_nodes=True, with_logits=False)
    n = case["n_nodes"].numpy()
    nan = torch.tensor(float("nan"), dtype=torch.bfloat16)
    for b in range(cfg.B):
        case["k_tree"][:, b, n[b]:] = nan
        case["v_tree"][:, b, n[b]:] = nan
    dcase = to_device(case)
    out, lse, bits, dense = gpu_attention(dcase)
    ref_out, ref_lse = oracle_attention(case_to_numpy(case), dense.cpu().numpy())
    assert_attention_close(out, lse, ref_out, ref_lse, f"M={N} D={D}")
    out2, lse2, _, _ = gpu_attention(dcase, simt=True)
    assert_attention_close(out2, lse2, ref_out, ref_lse, f"simt M={N} D={D}")


def _tree_case(parent, S, Hq, Hkv, d, Scap, seed, std=1.0):
    N = len(parent)
    cfg = CONFIGS[0].scaled(B=1, Hq=Hq, Hkv=Hkv, d=d, S_lo=S, S_hi=S, Scap=Scap, N=N, D=min(3, N - 1), std=std, V=0)
    case = make_case(cfg, seed=seed, with_logits=False)
    case["parent"] = torch.from_numpy(parent[None].astype(np.int32))
    return case


@pytest.mark.parametrize("S", [0, 1, 16, 200])
@pytest.mark.parametrize("d", [64, 128])
def test_closed_form_zero_keys_pins_the_visible_count(S, d):
    """K = 0 => lse = ln(S + depth + 1) and out = mean of the visible V rows."""
    rng = np.random.default_rng(S + d)
    parent = topk_expansion_tree(40, 6, 4, rng)
    case = _tree_case(parent, S, 4, 2, d, 256, seed=S)
    case["k_cache"].zero_()
    case["k_tree"].zero_()
    out, lse, bits, dense = gpu_attention(to_device(case))
    ref_out, ref_lse = oracle_attention(case_to_numpy(case), dense.cpu().numpy())
    vis = dense.cpu().numpy()[0, 0]
    want = np.log(S + vis.sum(1))
    assert np.abs(f32(lse)[0] - want[None, :]).max() < 1e-4
    assert np.abs(ref_lse[0] - want[None, :]).max() < 1e-12
    assert_attention_close(out, lse, ref_out, ref_lse, "zero keys")


@pytest.mark.parametrize("S", [0, 1, 16])
def test_leak_canary_one_hot_values(S):
    """Tree V rows are 100 * e_j and tree keys score alike, so a leaked
    non-ancestor or a missing ancestor moves the output by far more than 2e-2."""
    rng = np.random.default_rng(40 + S)
    N, d = 60, 64
    parent = topk_expansion_tree(N, 6, 10, rng)
    case = _tree_case(parent, S, 2, 1, d, 64, seed=S + 9)
    case["v_tree"].zero_()
    for j in range(N):
        case["v_tree"][0, 0, j, 0, j % d] = 100.0
    case["v_cache"].zero_()
    case["k_tree"].zero_()
    case["k_cache"].zero_()
    out, lse, bits, dense = gpu_attention(to_device(case))
    ref_out, ref_lse = oracle_attention(case_to_numpy(case), dense.cpu().numpy())
    vis = dense.cpu().numpy()[0, 0].astype(np.float64)
    want = np.zeros((N, d))
    for i in range(N):
        for j in np.flatnonzero(vis[i]):
            want[i, j % d] += 100.0 / (S + vis[i].sum())
    assert np.abs(ref_out[0, :, 0] - want).max() < 1e-9
    got = f32(out)[0]
    for h in range(2):
        assert np.abs(got[:, h] - want).max() <= 0.26      # 100/k rounded to bf16: half-ulp of 64..128 is 0.25
    # a leak of one key would shift some entry by >= 100/(S+8) > 4


MOVES = [
    # name, S, N, index of the dominant key (prefix row, or S + tree node)
    ("ragged_prefix_tile_second_half", 242, 8, 200),
    ("first_tile_of_the_item_second_half", 100, 8, 80),
    ("tree_tile_second_half", 40, 128, 40 + 100),
    ("whole_tile_then_ragged_tile", 370, 8, 340),
    # full, unmasked prefix tiles: the fast path's row-sum check has to reject the tile and the careful path redo it
    ("full_tile_first_half", 600, 8, 260),
    ("full_tile_second_half", 600, 8, 350),
    ("opening_tile_early_key", 600, 8, 5),
    ("opening_tile_late_key", 600, 8, 120),
    ("last_full_tile_last_key", 640, 8, 639),
    # a jump of about 2^367: 2^x overflows in the fast path, the factor of the rescale underflows to zero
    ("extreme_jump_in_a_full_tile", 600, 8, 350),
    ("extreme_jump_in_the_tree_tile", 40, 128, 40 + 100),
]


@pytest.mark.parametrize("name,S,N,big", MOVES, ids=[m[0] for m in MOVES])
@pytest.mark.parametrize("d", [64, 128])
def test_reference_maximum_moving_inside_a_tile(name, S, N, big, d):
    """The softmax keeps a lazy reference maximum and rescales only when the maximum grows by more than 2^8.
    Masked key tiles are worked through in two halves of 64 keys; here one key in the SECOND half of such a
    tile scores 2^12 above everything before it, so the reference moves after the first half has already
    produced its probabilities: they have to move with it.  All other scores are 0, so every visible key
    before the dominant one has weight 1 and that one 2^12.2: the output is a known mixture."""
    parent = chain_tree(N)                          # node i sees nodes 0..i: tree key j is visible to rows >= j
    case = _tree_case(parent, S, 2, 1, d, 384 if S < 384 else 768, seed=S + N)
    case["k_cache"].zero_()
    case["k_tree"].zero_()
    case["q"].fill_(1.0)
    amp = 0.75 * (128 / d) ** 0.5                   # score = d * amp / sqrt(d); 12.24 in log2 units for both head dims
    if name.startswith("extreme"):
        amp *= 30.0
    if big < S:
        case["k_cache"][0, 0, 0, big] = amp
    else:
        case["k_tree"][0, 0, big - S, 0] = amp
    out, lse, bits, dense = gpu_attention(to_device(case))
    ref_out, ref_lse = oracle_attention(case_to_numpy(case), dense.cpu().numpy())
    assert_attention_close(out, lse, ref_out, ref_lse, name)
    # the oracle's rows that see the dominant key are that key's V row up to the 2^-12 share of the others
    cn = case_to_numpy(case)
    vbig = orc.decode_bf16(cn["v_cache"][0][0, 0, big] if big < S else cn["v_tree"][0][0, big - S, 0])
    rows = range(N) if big < S else range(big - S, N)
    for i in rows:
        assert np.abs(ref_out[0, i, 0] - vbig).max() < 0.5      # the other keys share less than 0.1 of the weight


def test_non_ancestor_perturbation_leaves_rows_bit_identical():
    rng = np.random.default_rng(5)
    parent = topk_expansion_tree(64, 7, 8, rng)
    case = _tree_case(parent, 300, 8, 2, 128, 512, seed=3, std=128 ** -0.5)
    dcase = to_device(case)
    out1, lse1, bits, dense = gpu_attention(dcase)
    vis = dense.cpu().numpy()[0, 0]
    victim = 63
    dcase["k_tree"][0, 0, victim] = 30.0
    dcase["v_tree"][0, 0, victim] = -50.0
    out2, lse2, _, _ = gpu_attention(dcase)
    a, b = bf16_bits(out1), bf16_bits(out2)
    unaffected = np.flatnonzero(vis[:, victim] == 0)
    assert len(unaffected) >= 50
    assert np.array_equal(a[0, unaffected], b[0, unaffected])
    assert np.array_equal(f32(lse1)[0][:, unaffected], f32(lse2)[0][:, unaffected])
    assert not np.array_equal(a[0, victim], b[0, victim])


def test_state_safety_cache_and_inputs_are_not_written():
    cfg = CONFIGS[2].scaled(B=2, Hq=8, Hkv=2, S_lo=200, S_hi=400, Scap=512)
    dcase = to_device(make_case(cfg, seed=8, with_logits=False))
    before = {k: dcase[k].clone() for k in ("k_cache", "v_cache", "k_tree", "v_tree", "q", "prefix_len")}
    gpu_attention(dcase)
    for k, v in before.items():
        assert torch.equal(v, dcase[k]), f"{k} was modified by tree_verify_attn"


def test_chain_tree_is_causal_attention_and_one_node_is_decode():
    for N in (1, 37):
        case = _tree_case(chain_tree(N), 150, 4, 4, 128, 256, seed=N, std=0.3)
        out, lse, bits, dense = gpu_attention(to_device(case))
        cn = case_to_numpy(case)
        q = torch.from_numpy(orc.decode_bf16(cn["q"][0]))[0].permute(1, 0, 2)
        k = torch.cat([torch.from_numpy(orc.decode_bf16(cn["k_cache"][0]))[0, :, :150],
                       torch.from_numpy(orc.decode_bf16(cn["k_tree"][0]))[0].permute(1, 0, 2)], 1)
        v = torch.cat([torch.from_numpy(orc.decode_bf16(cn["v_cache"][0]))[0, :, :150],
                       torch.from_numpy(orc.decode_bf16(cn["v_tree"][0]))[0].permute(1, 0, 2)], 1)
        allow = torch.ones(N, 150 + N).tril(diagonal=150).bool()
        ref = torch.nn.functional.scaled_dot_product_attention(q, k, v, attn_mask=allow, scale=128 ** -0.5)
        err = np.abs(f32(out)[0] - ref.permute(1, 0, 2).numpy()).max()
        assert err <= ATTN_ATOL


def test_repeated_launches_are_bit_reproducible_and_never_time_out():
    """Units cut between CTAs are merged by whichever piece finishes last; the result must not depend on
    that order, and the bounded waits must never expire (they once did when a wait could lag two barrier
    phases behind)."""
    cfg = CONFIGS[4].scaled(L=1, V=0)
    dcase = make_case(cfg, seed=4001, device="cuda", with_logits=False)
    B, N = cfg.B, cfg.N
    bits = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(dcase["parent"], dcase["n_nodes"], N - 1, 1, bits, status)
    ws = torch.zeros(tv.tv_attn_workspace_bytes(B, N, cfg.Hq, cfg.Hkv, cfg.d, cfg.Scap), dtype=torch.uint8, device="cuda")
    first = None
    for it in range(60):
        out = torch.zeros(B, N, cfg.Hq, cfg.d, dtype=torch.bfloat16, device="cuda")
        lse = torch.zeros(B, cfg.Hq, N, dtype=torch.float32, device="cuda")
        tv.tree_verify_attn(dcase["q"][0], dcase["k_cache"][0], dcase["v_cache"][0], dcase["k_tree"][0],
                            dcase["v_tree"][0], dcase["prefix_len"], dcase["n_nodes"], bits, cfg.d ** -0.5, out,
                            ws, status, lse=lse)
        torch.cuda.synchronize()
        assert (status == 0).all(), f"launch {it}: status {status.cpu().tolist()}"
        if first is None:
            first = (out, lse)
        else:
            assert torch.equal(out, first[0]) and torch.equal(lse, first[1]), f"launch {it} differs from launch 0"


def test_back_to_back_launches_on_one_workspace_match_isolated_launches():
    """The layers of a step are launched back to back on one stream and one workspace, and a launch may
    start while the one in front is still draining.  Every launch must give exactly what it gives alone:
    no partial, counter or output of a neighbouring launch may leak in."""
    cfg = CONFIGS[4].scaled(L=4, B=6, V=0)
    dcase = make_case(cfg, seed=4100, device="cuda", with_logits=False)
    B, N, L = cfg.B, cfg.N, cfg.L
    bits = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(dcase["parent"], dcase["n_nodes"], N - 1, 1, bits, status)
    nbytes = tv.tv_attn_workspace_bytes(B, N, cfg.Hq, cfg.Hkv, cfg.d, cfg.Scap)
    ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")

    def launch(layer, out, lse, workspace):
        tv.tree_verify_attn(dcase["q"][layer], dcase["k_cache"][layer], dcase["v_cache"][layer],
                            dcase["k_tree"][layer], dcase["v_tree"][layer], dcase["prefix_len"], dcase["n_nodes"],
                            bits, cfg.d ** -0.5, out, workspace, status, lse=lse)

    alone = []
    for layer in range(L):                      # isolated: own workspace, synchronised on both sides
        out = torch.zeros(B, N, cfg.Hq, cfg.d, dtype=torch.bfloat16, device="cuda")
        lse = torch.zeros(B, cfg.Hq, N, dtype=torch.float32, device="cuda")
        launch(layer, out, lse, torch.zeros(nbytes, dtype=torch.uint8, device="cuda"))
        torch.cuda.synchronize()
        alone.append((out, lse))
    for rep in range(5):                        # back to back, 3 rounds over the layers, nothing in between
        outs = [torch.zeros(B, N, cfg.Hq, cfg.d, dtype=torch.bfloat16, device="cuda") for _ in range(3 * L)]
        lses = [torch.zeros(B, cfg.Hq, N, dtype=torch.float32, device="cuda") for _ in range(3 * L)]
        torch.cuda.synchronize()
        for i in range(3 * L):
            launch(i % L, outs[i], lses[i], ws)
        torch.cuda.synchronize()
        assert (status == 0).all(), f"status {status.cpu().tolist()}"
        for i in range(3 * L):
            assert torch.equal(outs[i], alone[i % L][0]) and torch.equal(lses[i], alone[i % L][1]), \
                f"round {rep}, launch {i} (layer {i % L}) differs from the isolated launch"


FULL = [(1, [(0, 0), (0, 17), (0, 31)]), (2, [(0, 0), (3, 5), (7, 7)]), (3, [(0, 0), (3, 7)]),
        (4, [(0, 0), (9, 3), (15, 7)])]


@pytest.mark.parametrize("ci,samples", FULL, ids=[CONFIGS[c].name for c, _ in FULL])
def test_attention_full_size_sampled_heads(ci, samples):
    """Full-size configs in the launch configuration the bench uses; the oracle
    checks sampled (sequence, KV head) slices one by one."""
    cfg = CONFIGS[ci].scaled(L=min(CONFIGS[ci].L, 2), V=0)
    dcase = make_case(cfg, seed=1000 * ci, device="cuda", with_logits=False)
    layer = cfg.L - 1
    out, lse, bits, dense = gpu_attention(dcase, layer)
    vis = dense.cpu().numpy()[:, 0]
    G = cfg.Hq // cfg.Hkv
    case_np = {k: (bf16_bits(v[layer:layer + 1]) if v.dtype == torch.bfloat16 else v.cpu().numpy())
               for k, v in dcase.items() if isinstance(v, torch.Tensor)}
    got_out, got_lse = f32(out), f32(lse)
    assert np.isfinite(got_out).all()
    for (b, hk) in samples:
        ref_out, ref_lse = oracle_attention_slice(case_np, 0, b, hk, G, vis, cfg.d ** -0.5)
        err = np.abs(got_out[b:b + 1, :, hk * G:(hk + 1) * G] - ref_out).max()
        assert err <= ATTN_ATOL, f"(b={b}, hk={hk}): {err}"
        assert np.abs(got_lse[b:b + 1, hk * G:(hk + 1) * G] - ref_lse).max() <= 2e-3


def test_layers_call_one_launch_many_layers_and_its_limits():
    """tree_verify_attn_layers: all layers in one launch (as many as the workspace has room for), against the
    oracle layer by layer; the same call as one launch per layer agrees to the rounding of the partials."""
    L = 35
    cfg = CONFIGS[0].scaled(B=3, L=L, S_lo=0, S_hi=600, Scap=640, N=15, Hq=8, Hkv=2, V=0)
    case = make_case(cfg, seed=77, ragged_nodes=True, with_logits=False)
    d = to_device(case)
    B, N, Hq, Hkv, dh = cfg.B, cfg.N, cfg.Hq, cfg.Hkv, cfg.d
    bits = torch.zeros(B, N, 1, dtype=torch.int32, device="cuda")
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(d["parent"], d["n_nodes"], N - 1, 1, bits, status)
    need = tv.tv_attn_workspace_bytes(B, N, Hq, Hkv, dh, cfg.Scap)
    ws = torch.zeros(need, dtype=torch.uint8, device="cuda")

    def run(flags, workspace):
        out = torch.full((L, B, N, Hq, dh), 3.0, dtype=torch.bfloat16, device="cuda")
        lse = torch.full((L, B, Hq, N), 3.0, dtype=torch.float32, device="cuda")
        n0 = tv.tv_launch_count()
        tv.tree_verify_attn_layers(d["q"], d["k_cache"], d["v_cache"], d["k_tree"], d["v_tree"], d["prefix_len"],
                                   d["n_nodes"], bits, dh ** -0.5, out, workspace, status, lse=lse, flags=flags)
        torch.cuda.synchronize()
        assert (status.cpu().numpy() == 0).all()
        return out, lse, tv.tv_launch_count() - n0

    out, lse, launches = run(tv.TV_ATTN_STABLE_INPUTS, ws)
    assert launches == 2                                    # the workspace has room for 32 layers
    vis = oracle_visibility(case["parent"], case["n_nodes"], bits_gpu=bits)
    cn = case_to_numpy(case)
    for l in range(L):
        ref_out, ref_lse = orc.tree_attention(cn["q"][l], cn["k_cache"][l], cn["v_cache"][l], cn["k_tree"][l],
                                              cn["v_tree"][l], cn["prefix_len"], cn["n_nodes"], vis[:, 0], dh ** -0.5)
        assert_attention_close(out[l], lse[l], ref_out, ref_lse, f"layer {l}")
    out2, lse2, launches2 = run(tv.TV_ATTN_LAUNCH_PER_LAYER, ws)
    assert launches2 == L
    assert (out.float() - out2.float()).abs().max().item() <= 2.0 ** -5
    # room for a single layer: still correct, one launch per layer
    per_layer = (B * Hkv * 2 * 8 + 255) // 256 * 256
    small = torch.zeros(need - 31 * per_layer, dtype=torch.uint8, device="cuda")
    out3, lse3, launches3 = run(0, small)
    assert launches3 == L and torch.equal(out3, out2) and torch.equal(lse3, lse2)
    with pytest.raises(tv.TreeVerifyError):                 # not even for one layer
        run(0, torch.zeros(need - 32 * per_layer, dtype=torch.uint8, device="cuda"))


def test_layers_call_with_padded_layer_strides_is_bit_equal_to_the_dense_call():
    """The layer strides are arguments of their own: tensors whose layers lie further apart than their size
    (a view into a larger allocation) give the same bits as dense ones."""
    L = 3
    cfg = CONFIGS[0].scaled(B=3, L=L, S_lo=0, S_hi=500, Scap=512, N=40, Hq=8, Hkv=2, d=128, V=0)
    case = to_device(make_case(cfg, seed=61, ragged_nodes=True, with_logits=False))
    B, N, Hq, Hkv, d, Scap = cfg.B, cfg.N, cfg.Hq, cfg.Hkv, cfg.d, cfg.Scap
    bits = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(case["parent"], case["n_nodes"], N - 1, 1, bits, st)
    ws = torch.zeros(tv.tv_attn_workspace_bytes(B, N, Hq, Hkv, d, Scap), dtype=torch.uint8, device="cuda")

    def padded(t, pad):
        per = t[0].numel()
        big = torch.full((L * (per + pad),), 7.0, dtype=t.dtype, device=t.device)
        v = torch.as_strided(big, t.shape, (per + pad,) + t[0].stride())
        v.copy_(t)
        return v

    def run(q, kc, vc, kt, vt, out):
        tv.tree_verify_attn_layers(q, kc, vc, kt, vt, case["prefix_len"], case["n_nodes"], bits, d ** -0.5, out, ws, st)
        torch.cuda.synchronize()
        assert (st.cpu().numpy() == 0).all()
        return out

    dense = run(case["q"], case["k_cache"], case["v_cache"], case["k_tree"], case["v_tree"],
                torch.zeros(L, B, N, Hq, d, dtype=torch.bfloat16, device="cuda"))
    out_p = padded(torch.zeros(L, B, N, Hq, d, dtype=torch.bfloat16, device="cuda"), 24)
    got = run(padded(case["q"], 8), padded(case["k_cache"], 4096), padded(case["v_cache"], 4096), padded(case["k_tree"], 16),
              padded(case["v_tree"], 16), out_p)
    assert torch.equal(got, dense)
    per = B * N * Hq * d                       # the gaps between the layers of the output were left alone
    gaps = torch.as_strided(out_p, (L, 24), (per + 24, 1), per)
    assert (gaps == 7.0).all()


@pytest.mark.parametrize("S", [700, 1100, 2600, 6000])
@pytest.mark.parametrize("G,d", [(2, 64), (4, 128)])
@pytest.mark.parametrize("B", [1, 3])
def test_units_cut_in_two_to_many_pieces(S, G, d, B):
    """Prefixes that are cut in two, three and more pieces (one KV head, few units): sums that stay in tensor memory
    between two pieces, and the flags of one and of several, twice with the same workspace contents."""
    cfg = CONFIGS[0].scaled(B=B, Hq=G, Hkv=1, d=d, S_lo=S - 130, S_hi=S, Scap=S + 200, N=40, D=6, V=0, tree="uniform")
    case = make_case(cfg, seed=S + G + B, ragged_nodes=True, with_logits=False)
    dcase = to_device(case)
    out, lse, bits, dense = gpu_attention(dcase)
    ref_out, ref_lse = oracle_attention(case_to_numpy(case), dense.cpu().numpy())
    assert_attention_close(out, lse, ref_out, ref_lse, f"S={S}")
    out2, lse2, _, _ = gpu_attention(dcase)
    assert torch.equal(out, out2) and torch.equal(lse, lse2)


CLUSTERS = [      # B, Hkv, G, N, S, d: units shared by 8, 4 and 2 CTAs; fewer key tiles than CTAs; one and two row tiles; padding
    (1, 1, 1, 1, 0, 64), (1, 2, 4, 17, 1, 128), (1, 8, 4, 17, 130, 128), (1, 8, 4, 33, 1000, 128), (2, 8, 3, 60, 900, 128),
    (1, 32, 1, 60, 1300, 128), (3, 4, 8, 40, 513, 64), (1, 64, 1, 9, 700, 128), (1, 5, 4, 200, 777, 128), (8, 8, 1, 256, 300, 64),
    (1, 1, 128, 5, 600, 128), (1, 1, 4, 60, 6200, 64),
]


@pytest.mark.parametrize("B,Hkv,G,N,S,d", CLUSTERS)
def test_units_shared_by_a_cluster(B, Hkv, G, N, S, d):
    cfg = CONFIGS[0].scaled(B=B, Hq=G * Hkv, Hkv=Hkv, d=d, S_lo=S // 3 if B > 1 else S, S_hi=S, Scap=S + N + 40, N=N,
                            D=min(6, N - 1), V=0, tree="uniform")
    case = make_case(cfg, seed=S + G + N, ragged_nodes=True, with_logits=False)
    dcase = to_device(case)
    for b in range(B):                       # rows behind the prefix hold NaN: nothing of them may reach an output
        dcase["k_cache"][0, b, :, int(case["prefix_len"][b]):] = float("nan")
        dcase["v_cache"][0, b, :, int(case["prefix_len"][b]):] = float("nan")
    out, lse, bits, dense = gpu_attention(dcase)
    ref_out, ref_lse = oracle_attention(case_to_numpy(case), dense.cpu().numpy())
    assert_attention_close(out, lse, ref_out, ref_lse, "cluster")
    out2, lse2, _, _ = gpu_attention(dcase)
    assert torch.equal(out, out2) and torch.equal(lse, lse2)


@pytest.mark.parametrize("N", [65, 129])
def test_last_row_tile_in_a_launch_of_its_own(N):
    """Odd numbers of row tiles (three and five) on enough key tiles: two launches, equal to the one-launch calls of the
    single layers up to the rounding of the partials and to the oracle on sampled heads."""
    cfg = CONFIGS[0].scaled(B=10, L=4, Hq=32, Hkv=8, d=64, S_lo=20, S_hi=400, Scap=4096, N=N, D=6, V=0, tree="uniform")
    case = make_case(cfg, seed=N, device="cuda", ragged_nodes=True, with_logits=False)
    B, L, Hq, Hkv, d = cfg.B, cfg.L, cfg.Hq, cfg.Hkv, cfg.d
    bits = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(case["parent"], case["n_nodes"], N - 1, 1, bits, st)
    ws = torch.zeros(tv.tv_attn_workspace_bytes(B, N, Hq, Hkv, d, cfg.Scap), dtype=torch.uint8, device="cuda")

    def run(flags):
        out = torch.full((L, B, N, Hq, d), 3.0, dtype=torch.bfloat16, device="cuda")
        lse = torch.full((L, B, Hq, N), 3.0, dtype=torch.float32, device="cuda")
        n0 = tv.tv_launch_count()
        tv.tree_verify_attn_layers(case["q"], case["k_cache"], case["v_cache"], case["k_tree"], case["v_tree"],
                                   case["prefix_len"], case["n_nodes"], bits, d ** -0.5, out, ws, st, lse=lse, flags=flags)
        torch.cuda.synchronize()
        return out, lse, tv.tv_launch_count() - n0

    out, lse, launches = run(0)
    one, _, per_layer = run(tv.TV_ATTN_LAUNCH_PER_LAYER)
    assert launches == 2 and per_layer == L and (st == 0).all()
    assert (out.float() - one.float()).abs().max().item() <= 2.0 ** -5
    cn = case_to_numpy(case)
    vis = oracle_visibility(case["parent"], case["n_nodes"], bits_gpu=bits)[:, 0]
    G = Hq // Hkv
    for l, b, hk in ((0, 0, 0), (1, 4, 3), (3, 9, 7)):
        ref_out, ref_lse = oracle_attention_slice(cn, l, b, hk, G, vis, d ** -0.5)
        assert_attention_close(out[l][b:b + 1, :, hk * G:(hk + 1) * G], lse[l][b:b + 1, hk * G:(hk + 1) * G], ref_out, ref_lse,
                               f"{l} {b} {hk}")


@pytest.mark.parametrize("G,N,d", [(2, 40, 64), (4, 40, 64), (2, 40, 128), (4, 40, 128)])
@pytest.mark.parametrize("longest", [900, 1400, 2100, 2800, 6000])
def test_long_unit_among_many_is_cut_in_many_pieces(G, N, d, longest):
    """Too many units for clusters, one of them far longer than the rest: its pieces are two, several and many, next to
    whole units of one to three key tiles; one and two row tiles, both head widths."""
    cfg = CONFIGS[0].scaled(B=80, Hq=G, Hkv=1, d=d, S_lo=0, S_hi=260, Scap=longest + 64, N=N, D=6, V=0, tree="uniform")
    case = make_case(cfg, seed=longest + G + d, ragged_nodes=True, with_logits=False)
    case["prefix_len"][33] = longest
    dcase = to_device(case)
    out, lse, bits, dense = gpu_attention(dcase)
    ref_out, ref_lse = oracle_attention(case_to_numpy(case), dense.cpu().numpy())
    assert_attention_close(out, lse, ref_out, ref_lse, f"longest={longest}")
    out2, lse2, _, _ = gpu_attention(dcase)
    assert torch.equal(out, out2) and torch.equal(lse, lse2)


@pytest.mark.parametrize("G,N,d", [(2, 40, 64), (4, 40, 64), (2, 40, 128), (4, 40, 128)])
def test_lengths_that_change_under_the_waiting_launch(G, N, d):
    """The tile table is built from the lengths a launch finds before the kernel in front is done, and again when they have
    changed: by a switch that makes every guess one key tile too long, and by a kernel in front that writes them."""
    cfg = CONFIGS[0].scaled(B=80, Hq=G, Hkv=1, d=d, S_lo=0, S_hi=700, Scap=1400, N=N, D=6, V=0, tree="uniform")
    case = make_case(cfg, seed=91 + G + d, ragged_nodes=True, with_logits=False)
    dcase = to_device(case)
    out, lse, bits, dense = gpu_attention(dcase)
    ref_out, ref_lse = oracle_attention(case_to_numpy(case), dense.cpu().numpy())
    assert_attention_close(out, lse, ref_out, ref_lse, "settled lengths")
    ws = torch.zeros(tv.tv_attn_workspace_bytes(80, N, G, 1, d, 1400), dtype=torch.uint8, device="cuda")
    status = torch.zeros(80, dtype=torch.int32, device="cuda")
    args = (dcase["q"][0], dcase["k_cache"][0], dcase["v_cache"][0], dcase["k_tree"][0], dcase["v_tree"][0])
    got, got_lse = torch.zeros_like(out), torch.zeros_like(lse)
    tv.tv_debug_attn_expire(*args, dcase["prefix_len"], dcase["n_nodes"], bits, d ** -0.5, got, ws, status, 2_000_000_000, 8,
                            lse=got_lse)
    assert torch.equal(got, out) and torch.equal(got_lse, lse)
    lengths = torch.zeros_like(dcase["prefix_len"])
    for other in (0, 1400, 333):
        lengths.fill_(other)
        tv.tree_verify_attn(*args, lengths, dcase["n_nodes"], bits, d ** -0.5, got, ws, status, lse=got_lse)
        lengths.copy_(dcase["prefix_len"])
        tv.tree_verify_attn(*args, lengths, dcase["n_nodes"], bits, d ** -0.5, got, ws, status, lse=got_lse)
        assert torch.equal(got, out) and torch.equal(got_lse, lse), other
    assert not status.any()


ODD = [(65, 64, False), (65, 128, True), (129, 64, True), (129, 128, False)]      # N, d, paged: three and five row tiles of G = 4


@pytest.mark.parametrize("N,d,paged", ODD)
@pytest.mark.parametrize("what", ["short", "below", "at", "long", "last beside", "first behind"])
def test_last_row_tile_goes_by_the_lengths_and_not_by_the_capacity(N, d, paged, what):
    """A cache that could hold enough key tiles for two launches.  With short prefixes and one key tile below the bound the call gives
    the bits it gives in a small cache, where it is one launch; at the bound the last row tile is cut elsewhere, and its bits are
    others; the oracle's values on sampled heads all the same, far beyond the bound, and where the second launch runs behind the first
    one instead of beside it."""
    B, L, Hkv, G, cap = 10, 4, 8, 4, 6400
    TT = (N + 127) // 128
    cfg = CONFIGS[0].scaled(B=B, L=L, Hq=G * Hkv, Hkv=Hkv, d=d, S_lo=20, S_hi=400, Scap=cap, N=N, D=6, V=0, tree="uniform")
    case = make_case(cfg, seed=N + d, device="cuda", ragged_nodes=True, with_logits=False)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if what != "short":
        bound = -(-12 * sms // (L * Hkv))                  # key tiles of the sequences together at which the rule changes
        behind = -(-(60 if d == 64 else 100) * sms // (L * Hkv))
        total = {"below": bound - 1, "at": bound, "long": bound + 120, "last beside": behind - 1, "first behind": behind}[what]
        tiles = np.full(B, total // B) + (np.arange(B) < total % B)
        tiles[0] -= 3
        tiles[1] += 3
        rows = (tiles - TT) * 128 - np.random.default_rng(N).integers(0, 128, B)
        assert rows.max() <= cap and rows.min() > 0
        case["prefix_len"] = torch.from_numpy(rows.astype(np.int32)).cuda()
    bits = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(case["parent"], case["n_nodes"], N - 1, 1, bits, st)
    ws = torch.zeros(tv.tv_attn_workspace_bytes(B, N, cfg.Hq, Hkv, d, cap), dtype=torch.uint8, device="cuda")

    def run(rows):
        out = torch.full((L, B, N, cfg.Hq, d), 3.0, dtype=torch.bfloat16, device="cuda")
        lse = torch.full((L, B, cfg.Hq, N), 3.0, dtype=torch.float32, device="cuda")
        kc, vc = (case[k][:, :, :, :rows].contiguous() for k in ("k_cache", "v_cache"))
        n0 = tv.tv_launch_count()
        if paged:
            kp, vp = (t.reshape(L, B, Hkv, rows // 128, 128, d).transpose(2, 3).reshape(L, -1, Hkv, 128, d).contiguous() for t in (kc, vc))
            table = torch.arange(B * (rows // 128), dtype=torch.int32, device="cuda").view(B, -1)
            tv.tree_verify_attn_paged_layers(case["q"], kp, vp, table, case["k_tree"], case["v_tree"], case["prefix_len"],
                                             case["n_nodes"], bits, d ** -0.5, out, ws, st, lse=lse)
        else:
            tv.tree_verify_attn_layers(case["q"], kc, vc, case["k_tree"], case["v_tree"], case["prefix_len"], case["n_nodes"],
                                       bits, d ** -0.5, out, ws, st, lse=lse)
        launches = tv.tv_launch_count() - n0
        torch.cuda.synchronize()
        assert (st == 0).all()
        return out, lse, launches

    out, lse, launches = run(cap)
    assert launches == 2
    if what in ("short", "below", "at"):
        small, small_lse, launches = run(1024)
        assert launches == 1 and torch.equal(out, small) == (what != "at")
        assert what == "at" or torch.equal(lse, small_lse)
    again, again_lse, _ = run(cap)
    assert torch.equal(out, again) and torch.equal(lse, again_lse)
    cn = case_to_numpy(case)
    vis = oracle_visibility(case["parent"], case["n_nodes"], bits_gpu=bits)[:, 0]
    for l, b, hk in ((0, 0, 0), (L - 1, 1, 7), (L // 2, 9, 3)):
        ref_out, ref_lse = oracle_attention_slice(cn, l, b, hk, G, vis, d ** -0.5)
        assert_attention_close(out[l][b:b + 1, :, hk * G:(hk + 1) * G], lse[l][b:b + 1, hk * G:(hk + 1) * G], ref_out, ref_lse,
                               f"{l} {b} {hk}")


@pytest.mark.parametrize("N,d", [(65, 64), (129, 128)])
@pytest.mark.parametrize("cap,launches", [(59, 1), (60, 2)])
def test_caches_without_room_for_long_work_have_one_launch(N, d, cap, launches):
    """Short prefixes in a cache of one key tile per SM less than two launches need, and in one that allows them: the second one
    is made only there, and the results are the same bits."""
    B, L, Hkv, G = 4, 2, 2, 4
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = (-(-cap * sms // (B * L * Hkv)) - (N + 127) // 128) * 128
    cfg = CONFIGS[0].scaled(B=B, L=L, Hq=G * Hkv, Hkv=Hkv, d=d, S_lo=200, S_hi=900, Scap=1024, N=N, D=6, V=0, tree="uniform")
    case = make_case(cfg, seed=N, device="cuda", ragged_nodes=True, with_logits=False)
    bits = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(case["parent"], case["n_nodes"], N - 1, 1, bits, st)
    ws = torch.zeros(tv.tv_attn_workspace_bytes(B, N, cfg.Hq, Hkv, d, rows), dtype=torch.uint8, device="cuda")

    def run(rows):
        kc, vc = (torch.full((L, B, Hkv, rows, d), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in "kv")
        kc[:, :, :, :900], vc[:, :, :, :900] = case["k_cache"][:, :, :, :900], case["v_cache"][:, :, :, :900]
        out = torch.full((L, B, N, cfg.Hq, d), 3.0, dtype=torch.bfloat16, device="cuda")
        n0 = tv.tv_launch_count()
        tv.tree_verify_attn_layers(case["q"], kc, vc, case["k_tree"], case["v_tree"], case["prefix_len"], case["n_nodes"], bits,
                                   d ** -0.5, out, ws, st)
        torch.cuda.synchronize()
        return out, tv.tv_launch_count() - n0

    out, n = run(rows)
    assert n == launches
    other, n = run(rows // 2)
    assert n == 1 and torch.equal(out, other) and not st.any()


def torch_attention_slice(case, l, b, h, hk, vis, scale):
    """One query head in fp32: (out [N,d], lse [N]) of the rows that have a node."""
    S, n = int(case["prefix_len"][b]), int(case["n_nodes"][b])
    k, v = (torch.cat([case[c][l][b, hk, :S], case[t][l][b, :n, hk]]).float() for c, t in (("k_cache", "k_tree"), ("v_cache", "v_tree")))
    s = case["q"][l][b, :n, h].float() @ k.T * scale
    s[:, S:] += torch.where(torch.from_numpy(vis[b, :n, :n]).cuda() != 0, 0.0, float("-inf"))
    return torch.softmax(s, -1) @ v, torch.logsumexp(s, -1)


@pytest.mark.parametrize("N,G,d", [(145, 32, 64), (149, 64, 128), (149, 128, 64)])      # 37, 75 and 149 row tiles
@pytest.mark.parametrize("what", ["below", "at", "long"])
def test_wide_head_groups_have_the_last_row_tile_behind_the_others(N, G, d, what):
    """With lengths just below the bound the call gives the bits it gives in a cache that is too small for two launches; from the
    bound on the last row tile comes out of the second launch: fp32 values on heads at both ends."""
    B, L, Hkv, TT = 3, 4, 2, 2
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    bound = -(-60 * sms // (L * Hkv))                      # key tiles of the sequences together from which the work is split
    each = (bound - 1) // B                                # a cache of so many key tiles (the tree's among them) has one launch
    tiles = np.full(B, {"below": each, "at": bound // B, "long": bound // B + 40}[what])
    if what == "at":
        tiles[:bound % B] += 1
    cap = (each - TT) * 128
    big = (bound // B + 60) * 128
    cfg = CONFIGS[0].scaled(B=B, L=L, Hq=G * Hkv, Hkv=Hkv, d=d, S_lo=cap, S_hi=cap, Scap=big, N=N, D=6, V=0, tree="uniform")
    case = make_case(cfg, seed=N + G, device="cuda", ragged_nodes=True, with_logits=False)
    case["prefix_len"] = torch.from_numpy(((tiles - TT) * 128).astype(np.int32)).cuda()
    case["n_nodes"][0] = N
    bits = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(case["parent"], case["n_nodes"], N - 1, 1, bits, st)
    ws = torch.zeros(tv.tv_attn_workspace_bytes(B, N, cfg.Hq, Hkv, d, big), dtype=torch.uint8, device="cuda")

    def run(rows):
        out = torch.full((L, B, N, cfg.Hq, d), 3.0, dtype=torch.bfloat16, device="cuda")
        lse = torch.full((L, B, cfg.Hq, N), 3.0, dtype=torch.float32, device="cuda")
        kc, vc = (case[k] if rows == big else case[k][:, :, :, :rows].contiguous() for k in ("k_cache", "v_cache"))
        n0 = tv.tv_launch_count()
        tv.tree_verify_attn_layers(case["q"], kc, vc, case["k_tree"], case["v_tree"], case["prefix_len"], case["n_nodes"], bits,
                                   d ** -0.5, out, ws, st, lse=lse)
        torch.cuda.synchronize()
        assert not st.any()
        return out, lse, tv.tv_launch_count() - n0

    out, lse, launches = run(big)
    assert launches == 2
    again, again_lse, _ = run(big)
    assert torch.equal(out, again) and torch.equal(lse, again_lse)
    if what == "below":
        small, small_lse, launches = run(cap)
        assert launches == 1 and torch.equal(out, small) and torch.equal(lse, small_lse)
    vis = oracle_visibility(case["parent"], case["n_nodes"], bits_gpu=bits)[:, 0]
    for l, b, h in ((0, 0, 0), (L - 1, 1, cfg.Hq - 1), (1, 2, G)):
        want, want_lse = torch_attention_slice(case, l, b, h, h // G, vis, d ** -0.5)
        n = want.shape[0]
        assert (out[l][b, :n, h].float() - want).abs().max() <= ATTN_ATOL and not out[l][b, n:, h].any()
        assert (lse[l][b, h, :n] - want_lse).abs().max() <= 2e-3 and torch.isneginf(lse[l][b, h, n:]).all()


@pytest.mark.parametrize("N,d,G", [(65, 64, 4), (65, 128, 4), (129, 128, 4), (160, 64, 4), (44, 128, 8), (225, 64, 16)])
def test_last_row_tile_beside_the_others_keeps_the_order_of_the_stream(N, d, G):
    """The two launches of an odd last row tile run at the same time.  Inputs written by the kernels directly in front, outputs
    overwritten by the one directly behind, call after call, give the bits of a call with the device idle on either side, and so
    does a replayed graph; three, five and 29 row tiles, the last one full, short and nearly empty."""
    B, Hkv, cap = 14, 8, 10240
    cfg = CONFIGS[0].scaled(B=B, L=1, Hq=G * Hkv, Hkv=Hkv, d=d, S_lo=2600, S_hi=4300, Scap=cap, N=N, D=6, V=0, tree="uniform")
    cases = [make_case(cfg, seed=N + d + x, device="cuda", ragged_nodes=True, with_logits=False) for x in (0, 1)]
    names = ("q", "prefix_len", "n_nodes", "parent")
    here = {k: torch.empty_like(cases[0][k]) for k in names}
    bits = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    ws = torch.zeros(tv.tv_attn_workspace_bytes(B, N, cfg.Hq, Hkv, d, cap), dtype=torch.uint8, device="cuda")
    out = torch.zeros(B, N, cfg.Hq, d, dtype=torch.bfloat16, device="cuda")
    kept = torch.zeros(2, *out.shape, dtype=torch.bfloat16, device="cuda")
    c = cases[0]

    def step(x, idle):
        for k in names:
            here[k].copy_(cases[x][k])
        tv.tree_build_mask(here["parent"], here["n_nodes"], N - 1, 1, bits, st)
        idle()
        tv.tree_verify_attn(here["q"][0], c["k_cache"][0], c["v_cache"][0], c["k_tree"][0], c["v_tree"][0], here["prefix_len"],
                            here["n_nodes"], bits, d ** -0.5, out, ws, st)
        idle()
        kept[x].copy_(out)
        out.fill_(7.0)

    n0 = tv.tv_launch_count()
    for x in (0, 1):
        step(x, torch.cuda.synchronize)
    assert tv.tv_launch_count() - n0 == 6                     # mask and two attention launches each
    want = kept.clone()
    for _ in range(4):
        for x in (0, 1):
            step(x, lambda: None)
        torch.cuda.synchronize()
        assert torch.equal(kept, want)
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(stream), torch.cuda.graph(graph):
        for x in (0, 1):
            step(x, lambda: None)
    for _ in range(3):
        kept.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(kept, want)
    assert not st.any()
    vis = oracle_visibility(cases[0]["parent"], cases[0]["n_nodes"])[:, 0]
    cn = case_to_numpy(cases[0])
    for b, hk in ((0, 0), (B - 1, 7)):
        ref_out, ref_lse = oracle_attention_slice(cn, 0, b, hk, G, vis, d ** -0.5)
        assert np.abs(want[0][b:b + 1, :, hk * G:(hk + 1) * G].float().cpu().numpy() - ref_out).max() <= 2e-2


@pytest.mark.parametrize("N,d,in_cache", [(65, 64, False), (65, 128, True), (129, 128, False), (129, 64, True)])
def test_pairs_of_launches_behind_one_another(N, d, in_cache):
    """Three pairs of launches in a row on one workspace, as one call with room for a layer a launch and as three calls: nothing in
    between, each second launch letting the next pair go while its first one runs.  The bits of each layer on its own with the device
    idle on either side, eagerly and from a graph; a tree that does not fit its cache is reported beside them."""
    B, Hkv, G, cap, L = 14, 8, 4, 10240, 3
    cfg = CONFIGS[0].scaled(B=B, L=L, Hq=G * Hkv, Hkv=Hkv, d=d, S_lo=2600, S_hi=4300, Scap=cap, N=N, D=6, V=0, tree="uniform")
    c = make_case(cfg, seed=N + d, device="cuda", ragged_nodes=True, with_logits=False)
    full = 5 if in_cache else B                            # this sequence has no room for its tree
    if in_cache:
        c["prefix_len"][full] = cap
        for b in range(B):
            S, n = int(c["prefix_len"][b]), min(N, cap - int(c["prefix_len"][b]))
            for k, t in (("k_cache", "k_tree"), ("v_cache", "v_tree")):
                c[k][:, b, :, S:S + n] = c[t][:, b, :n].transpose(1, 2)
    keep = [b for b in range(B) if b != full]
    kt, vt = (None, None) if in_cache else (c["k_tree"], c["v_tree"])
    bits = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    room = tv.tv_attn_workspace_bytes(B, N, cfg.Hq, Hkv, d, cap)
    NP = ((N + 31) // 32 + 1) // 2
    ws = torch.zeros(room - 31 * ((B * Hkv * NP * 16 + 255) // 256 * 256), dtype=torch.uint8, device="cuda")

    def run(one_call, idle):
        out = torch.full((L, B, N, cfg.Hq, d), 3.0, dtype=torch.bfloat16, device="cuda")
        n0 = tv.tv_launch_count()
        tv.tree_build_mask(c["parent"], c["n_nodes"], N - 1, 1, bits, st)
        idle()
        if one_call:
            tv.tree_verify_attn_layers(c["q"], c["k_cache"], c["v_cache"], kt, vt, c["prefix_len"], c["n_nodes"], bits, d ** -0.5,
                                       out, ws, st, flags=tv.TV_ATTN_STABLE_INPUTS)
        for l in () if one_call else range(L):
            tv.tree_verify_attn(c["q"][l], c["k_cache"][l], c["v_cache"][l], None if kt is None else kt[l], None if vt is None else vt[l],
                                c["prefix_len"], c["n_nodes"], bits, d ** -0.5, out[l], ws, st)
            idle()
        assert tv.tv_launch_count() - n0 == 1 + 2 * L
        return out

    def check(out):
        torch.cuda.synchronize()
        assert torch.equal(out[:, keep], want) and st.tolist() == [tv.TV_ST_CAPACITY if b == full else 0 for b in range(B)]

    want = run(False, torch.cuda.synchronize)[:, keep]
    for _ in range(3):
        check(run(False, lambda: None))
        check(run(True, lambda: None))
    for one_call in (False, True):
        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.stream(stream), torch.cuda.graph(graph):
            out = run(one_call, lambda: None)
        for _ in range(3):
            out.zero_()
            graph.replay()
            check(out)
    cn = case_to_numpy(c)
    vis = oracle_visibility(c["parent"], c["n_nodes"], bits_gpu=bits)[:, 0]
    for l, b, hk in ((0, 0, 0), (L - 1, B - 1, 7)):
        ref_out, _ = oracle_attention_slice(cn, l, b, hk, G, vis, d ** -0.5)
        assert np.abs(want[l][keep.index(b), :, hk * G:(hk + 1) * G].float().cpu().numpy() - ref_out[0]).max() <= ATTN_ATOL


@pytest.mark.parametrize("N,d", [(65, 64), (129, 128)])
@pytest.mark.parametrize("S", [300, 4000])       # the second launch has nothing to do, its share
def test_last_row_tile_without_leave_to_start_waits_for_the_others(N, d, S):
    """The second of two launches that run at the same time goes by a flag of the first; where it does not find it (a switch holds it
    back) it waits, and the results are the same bits, in turn with calls that do find it on one workspace."""
    B, Hkv, G, cap = 14, 8, 4, 10240
    cfg = CONFIGS[0].scaled(B=B, L=1, Hq=G * Hkv, Hkv=Hkv, d=d, S_lo=S // 2, S_hi=S, Scap=cap, N=N, D=6, V=0, tree="uniform")
    c = make_case(cfg, seed=N, device="cuda", ragged_nodes=True, with_logits=False)
    bits = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(c["parent"], c["n_nodes"], N - 1, 1, bits, st)
    ws = torch.zeros(tv.tv_attn_workspace_bytes(B, N, cfg.Hq, Hkv, d, cap), dtype=torch.uint8, device="cuda")
    args = (c["q"][0], c["k_cache"][0], c["v_cache"][0], c["k_tree"][0], c["v_tree"][0], c["prefix_len"], c["n_nodes"], bits, d ** -0.5)
    want = torch.zeros(B, N, cfg.Hq, d, dtype=torch.bfloat16, device="cuda")
    tv.tree_verify_attn(*args, want, ws, st)
    for mode in (32, 0, 32, 32, 0):
        out = torch.full_like(want, 3.0)
        n0 = tv.tv_launch_count()
        tv.tv_debug_attn_expire(*args, out, ws, st, 2_000_000_000, mode)
        assert tv.tv_launch_count() - n0 == 2
        torch.cuda.synchronize()
        assert torch.equal(out, want) and not st.any()


@pytest.mark.parametrize("G,N,d", [(2, 40, 64), (4, 40, 64), (2, 40, 128), (4, 40, 128)])
@pytest.mark.parametrize("S,other", [(300, 300), (1024, 1024), (1025, 1025), (300, 100)])
def test_equal_units_stay_whole_while_they_are_short(S, other, G, N, d):
    """Fewer units than CTA groups, but more than half: of equal length up to eight prefix tiles (whole, one a group), one row
    beyond that and with one shorter unit (cut)."""
    cfg = CONFIGS[0].scaled(B=90, Hq=G, Hkv=1, d=d, S_lo=S, S_hi=S, Scap=S + 64, N=N, D=6, V=0, tree="uniform")
    case = make_case(cfg, seed=S + G + d + other, ragged_nodes=True, with_logits=False)
    case["prefix_len"][17] = other
    dcase = to_device(case)
    out, lse, bits, dense = gpu_attention(dcase)
    ref_out, ref_lse = oracle_attention(case_to_numpy(case), dense.cpu().numpy())
    assert_attention_close(out, lse, ref_out, ref_lse, f"S={S} {other}")
    out2, lse2, _, _ = gpu_attention(dcase)
    assert torch.equal(out, out2) and torch.equal(lse, lse2)


@pytest.mark.parametrize("B,Hkv,G,N,S,d", [(1, 2, 2, 15, 128, 64), (1, 8, 4, 17, 1000, 128), (1, 32, 1, 60, 1300, 128),
                                           (3, 4, 8, 40, 513, 64), (1, 5, 4, 200, 777, 128), (1, 1, 4, 60, 6200, 64)])
def test_cluster_partials_are_not_rounded(B, Hkv, G, N, S, d):
    """Zero keys: every weight is 1 and an output is a mean of values in [1, 2).  Units shared by a cluster give the bf16 rounding
    of the exact mean: partials in 32 bits leave an error of 2^-14 of it at most (2^-23 for each of the up to 500 sums of 16 keys),
    where partials rounded to bf16 (2^-8 each) miss the right rounding in one element of five."""
    cfg = CONFIGS[0].scaled(B=B, Hq=G * Hkv, Hkv=Hkv, d=d, S_lo=S, S_hi=S, Scap=S + 40, N=N, D=min(6, N - 1), V=0, tree="uniform")
    case = to_device(make_case(cfg, seed=S + G + N, with_logits=False))
    g = torch.Generator(device="cuda")
    g.manual_seed(S)
    for k in ("k_cache", "k_tree"):
        case[k].zero_()
    for k in ("v_cache", "v_tree"):
        case[k].copy_(torch.rand(case[k].shape, device="cuda", generator=g) * 0.98 + 1.0)
    out, _, _, dense = gpu_attention(case)
    vis = dense.reshape(B, N, N).cuda().double()
    tree = torch.einsum("bij,bjhd->bihd", vis, case["v_tree"][0].double())
    prefix = case["v_cache"][0][:, :, :S].double().sum(2)                       # [B, Hkv, d]
    exact = (tree + prefix[:, None]) / (S + vis.sum(-1))[:, :, None, None]      # [B, N, Hkv, d]
    exact = exact.repeat_interleave(G, dim=2)
    best = (exact.to(torch.bfloat16).double() - exact).abs()
    assert ((out.cuda().reshape(exact.shape).double() - exact).abs() <= best + 2.0 ** -14 * exact).all()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,Hkv,G,N,S", [(90, 1, 4, 20, 300), (90, 1, 4, 40, 700), (3, 1, 4, 20, 6000), (1, 2, 4, 20, 700), (1, 4, 8, 40, 1500)])
def test_nan_queries_and_keys_give_nan_rows(B, Hkv, G, N, S, d):
    """Whole units, units cut in pieces, clusters, one and two row tiles: a query with a NaN gives a NaN row (as does a key with a
    NaN to the rows that see it) and changes no bit of another row."""
    cfg = CONFIGS[0].scaled(B=B, Hq=G * Hkv, Hkv=Hkv, d=d, S_lo=S // 2 if B < 90 else S, S_hi=S, Scap=S + 20, N=N, D=6, V=0, tree="uniform")
    case = to_device(make_case(cfg, seed=S + B + d, with_logits=False))
    want, _, _, dense = gpu_attention(case)
    case["q"][0, :, 3, 0, 5] = float("nan")
    case["q"][0, B - 1, N - 1, :, :] = float("nan")
    case["k_tree"][0, 0, 2, 0, 7] = float("nan")
    out, _, _, _ = gpu_attention(case)
    bad = torch.zeros(B, N, G * Hkv, dtype=torch.bool, device="cuda")
    bad[:, 3, 0] = True
    bad[B - 1, N - 1] = True
    bad[0, :, :G] |= dense.reshape(B, N, N)[0, :, 2].bool().cuda()[:, None]
    assert torch.isnan(out[bad]).all()
    assert torch.equal(out[~bad], want[~bad])

"""Launch overlap between the kernels of a step (programmatic stream serialisation) must never let a kernel
read what the kernel in front is still writing, nor lose a status bit.

  - kv_commit directly followed by tree_verify_attn (no mask launch in between): the attention reads
    prefix_len before its own wait, so it must only start when the commit is complete;
  - tree_build_mask directly followed by a one-layer attention that raises a status bit itself (a tree
    that does not fit the cache in the in-cache layout; a page id outside the pool): the mask kernel stores
    status last, and the attention's bit must survive it.
All calls of a test go to one stream with no synchronisation in between, many times over."""
import numpy as np
import pytest
import torch

import paper_2603_08088_b200 as tv
from oracle import tree_verify_oracle as orc
from workloads import CONFIGS, make_case, case_to_numpy, bf16_bits
from gpu_util import to_device, f32, i32, assert_attention_close, oracle_visibility

pytestmark = pytest.mark.gpu


def test_attention_directly_behind_commit_sees_the_new_prefix():
    """A step, then at once another attention over the same tree with the mask of the step: its keys are the
    prefix as the commit left it.  The prefix lengths are chosen so that the committed rows open a new key
    tile (126 -> 134 rows) or fill the last one, and the values are N(0,1), so stale lengths or rows move
    the output by far more than the tolerance."""
    cfg = CONFIGS[2].scaled(B=6, Hq=8, Hkv=2, S_lo=126, S_hi=126, Scap=256, N=64, V=2048, std=1.0)
    for rep in range(6):
        case = make_case(cfg, seed=7700 + rep)
        case["prefix_len"][:] = torch.tensor([126, 127, 120, 1, 250 - 8, 128], dtype=torch.int32)
        d = to_device(case)
        P, Dp1 = case["retrieve"].shape[1], cfg.D + 1
        buf = tv.StepBuffers(cfg.L, cfg.B, cfg.N, cfg.Hq, cfg.Hkv, cfg.d, cfg.Scap, cfg.V, P, Dp1)
        out2 = torch.full((cfg.B, cfg.N, cfg.Hq, cfg.d), 3.0, dtype=torch.bfloat16, device="cuda")
        lse2 = torch.full((cfg.B, cfg.Hq, cfg.N), 3.0, dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        tv.verify_step(d, buf, cfg.d ** -0.5)            # mask, attention, accept, commit
        tv.tree_verify_attn(d["q"][0], d["k_cache"][0], d["v_cache"][0], d["k_tree"][0], d["v_tree"][0],
                            d["prefix_len"], d["n_nodes"], buf.anc_bits, cfg.d ** -0.5, out2, buf.attn_ws, buf.status,
                            lse=lse2)
        torch.cuda.synchronize()
        ref = orc.verify_step(case_to_numpy(case), cfg.d ** -0.5, use_given_retrieve=False)
        assert (ref["accept"]["accept_len"] == cfg.D).all()            # planted: every prefix grows by D + 1 rows
        assert np.array_equal(i32(d["prefix_len"]), ref["prefix_len"])
        assert (i32(buf.status) == 0).all()
        c = case_to_numpy(case)
        vis = oracle_visibility(case["parent"], case["n_nodes"])
        want, want_lse = orc.tree_attention(c["q"][0], ref["k_cache"][0], ref["v_cache"][0], c["k_tree"][0], c["v_tree"][0],
                                            ref["prefix_len"], c["n_nodes"], vis[:, 0], cfg.d ** -0.5)
        assert_attention_close(out2, lse2, want, want_lse, f"attention behind the commit, repetition {rep}")
        # the same rows over the old prefix are far away: the check above can tell the two apart
        old, _ = orc.tree_attention(c["q"][0], c["k_cache"][0], c["v_cache"][0], c["k_tree"][0], c["v_tree"][0],
                                    c["prefix_len"], c["n_nodes"], vis[:, 0], cfg.d ** -0.5)
        assert np.abs(old - want).max() > 0.2


def test_status_bits_raised_by_a_one_layer_attention_survive_the_mask_kernel():
    cfg = CONFIGS[0].scaled(B=2, S_lo=100, S_hi=100, Scap=128, N=15)
    case = make_case(cfg, seed=12, with_logits=False)
    g = to_device(case)
    B, N, Hq, Hkv, d = cfg.B, cfg.N, cfg.Hq, cfg.Hkv, cfg.d
    bits = torch.zeros(B, N, 1, dtype=torch.int32, device="cuda")
    ws = torch.zeros(max(256, tv.tv_attn_workspace_bytes(B, N, Hq, Hkv, d, cfg.Scap)), dtype=torch.uint8, device="cuda")
    out = torch.zeros(B, N, Hq, d, dtype=torch.bfloat16, device="cuda")
    # in-cache layout: 120 + 15 rows do not fit 128; 100 + 15 do
    S = torch.tensor([120, 100], dtype=torch.int32, device="cuda")
    # paged layout: one page per sequence, the second sequence names a page outside the pool of 3
    kp = torch.zeros(3, Hkv, 128, d, dtype=torch.bfloat16, device="cuda")
    bt = torch.tensor([[1], [3]], dtype=torch.int32, device="cuda")
    statuses = []
    for rep in range(40):
        st1 = torch.full((B,), 64, dtype=torch.int32, device="cuda")       # the mask call overwrites it
        tv.tree_build_mask(g["parent"], g["n_nodes"], N - 1, 1, bits, st1)
        tv.tree_verify_attn(g["q"][0], g["k_cache"][0], g["v_cache"][0], None, None, S, g["n_nodes"], bits, d ** -0.5,
                            out, ws, st1)
        st2 = torch.full((B,), 64, dtype=torch.int32, device="cuda")
        tv.tree_build_mask(g["parent"], g["n_nodes"], N - 1, 1, bits, st2)
        tv.tree_verify_attn_paged(g["q"][0], kp, kp, bt, g["k_tree"][0], g["v_tree"][0], g["prefix_len"], g["n_nodes"],
                                  bits, d ** -0.5, out, ws, st2)
        statuses.append((st1, st2))
    torch.cuda.synchronize()
    for rep, (st1, st2) in enumerate(statuses):
        assert i32(st1).tolist() == [tv.TV_ST_CAPACITY, 0], f"repetition {rep}: {i32(st1).tolist()}"
        assert i32(st2).tolist() == [0, tv.TV_ST_BAD_INDEX], f"repetition {rep}: {i32(st2).tolist()}"


@pytest.mark.parametrize("in_cache", [False, True])
@pytest.mark.parametrize("B,L,S,N,launches", [(1, 1, 1500, 33, 1), (12, 3, 2500, 33, 1), (12, 8, 2800, 65, 2)])
def test_scan_beside_the_attention_changes_nothing(B, L, S, N, launches, in_cache):
    """verify_step lets the vocabulary scan overlap the attention in front of it.  Three steps in a row without a
    synchronisation, each on the cache and the lengths the one before has left, give bit for bit what the same calls
    with the ordered tree_accept give (acceptance and commit wait for the attention in both).  One attention launch, and two that
    run at the same time, of which the second lets the scan go while the first still runs."""
    cfg = CONFIGS[2].scaled(B=B, L=L, Hq=16, Hkv=4, S_lo=S // 2, S_hi=S, Scap=S + 300, V=30001, N=N, D=6)
    case = to_device(make_case(cfg, seed=B + L))

    def steps(ordered):
        c = {k: (v.clone() if isinstance(v, torch.Tensor) else v) for k, v in case.items()}
        P, Dp1 = cfg.N, cfg.D + 1
        outs = []
        for _ in range(3):
            buf = tv.StepBuffers(L, B, cfg.N, cfg.Hq, cfg.Hkv, cfg.d, cfg.Scap, cfg.V, P, Dp1)
            if not ordered:
                tv.verify_step(c, buf, cfg.d ** -0.5, in_cache=in_cache)
            else:
                tv.tree_build_mask(c["parent"], c["n_nodes"], Dp1 - 1, P, buf.anc_bits, buf.status, depth=buf.depth,
                                   anc_table=buf.anc_table, retrieve_indices=buf.retrieve, n_paths=buf.n_paths)
                n0 = tv.tv_launch_count()
                tv.tree_verify_attn_layers(c["q"], c["k_cache"], c["v_cache"], None if in_cache else c["k_tree"],
                                           None if in_cache else c["v_tree"], c["prefix_len"], c["n_nodes"], buf.anc_bits,
                                           cfg.d ** -0.5, buf.out, buf.attn_ws, buf.status, flags=tv.TV_ATTN_STABLE_INPUTS)
                assert tv.tv_launch_count() - n0 == launches
                torch.cuda.synchronize()
                tv.tree_accept(c["logits"], c["tokens"], buf.retrieve, c["n_nodes"], buf.argmax_tok, buf.accept_len,
                               buf.best_path, buf.accepted_nodes, buf.next_token, buf.accept_ws, buf.status)
                if in_cache:
                    tv.kv_commit_inplace(c["k_cache"], c["v_cache"], buf.accepted_nodes, buf.accept_len, c["prefix_len"],
                                         cfg.N, buf.status)
                else:
                    tv.kv_commit(c["k_cache"], c["v_cache"], c["k_tree"], c["v_tree"], buf.accepted_nodes, buf.accept_len,
                                 c["prefix_len"], buf.status)
                torch.cuda.synchronize()
            outs.append((buf.out, buf.status, buf.argmax_tok, buf.accept_len, buf.accepted_nodes, buf.next_token))
        torch.cuda.synchronize()
        return [t for o in outs for t in o] + [c["k_cache"], c["v_cache"], c["prefix_len"]]

    for a, b in zip(steps(False), steps(True)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("B,N,V", [(1, 17, 30001), (2, 9, 1003), (8, 64, 128257)])
def test_scan_beside_the_attention_reads_what_the_logits_are_now(B, N, V):
    """Steps without a synchronisation on one logits and one token buffer that are rewritten between them, with an attention
    of few units in front (it leaves SMs to the scan at once): short scans and a long one, entries on both sides of the whole
    vectors of a row.  The argmax of every step is that of the logits of its own step."""
    cfg = CONFIGS[0].scaled(B=B, L=1, Hq=2, Hkv=1, d=64, S_lo=300, S_hi=300, Scap=1024, N=N, D=min(6, N - 1), V=V, tree="uniform")
    c = to_device(make_case(cfg, seed=V))
    g = torch.Generator(device="cuda")
    g.manual_seed(V)
    steps = 12
    logits = [torch.randn(B, N, V, device="cuda", generator=g).to(torch.bfloat16) for _ in range(steps)]
    ends = list(range(8)) + list(range(V - 8, V))
    for s, l in enumerate(logits):                       # half of the rows have their maximum at an end of the row
        for i in range(0, N, 2):
            l[:, i, ends[(5 * s + i) % 16]] = 16.0 + s
    tokens = [torch.randint(0, V, (B, N), dtype=torch.int32, device="cuda", generator=g) for _ in range(steps)]
    buf = [tv.StepBuffers(1, B, N, cfg.Hq, cfg.Hkv, cfg.d, cfg.Scap, V, N, cfg.D + 1) for _ in range(steps)]
    seen = torch.zeros(steps, B, N, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    for s in range(steps):
        c["logits"].copy_(logits[s])
        torch.add(tokens[s], 0, out=c["tokens"])
        tv.verify_step(c, buf[s], cfg.d ** -0.5)
        seen[s].copy_(buf[s].argmax_tok)
    torch.cuda.synchronize()
    for s in range(steps):
        l = logits[s].float()
        first = torch.where(l == l.amax(-1, keepdim=True), torch.arange(V, device="cuda"), V).amin(-1)
        assert torch.equal(seen[s].long(), first), s
        ref = orc.greedy_accept(i32(buf[s].retrieve), i32(tokens[s]), i32(c["n_nodes"]), i32(seen[s]))
        for k in ("accept_len", "accepted_nodes", "next_token"):
            assert np.array_equal(i32(getattr(buf[s], k)), ref[k]), (s, k)


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("B,Hkv,G", [(80, 1, 4), (2, 2, 4)])      # the even cut, the cluster kernel
def test_early_reads_see_lengths_and_pages_rewritten_in_place(B, Hkv, G, paged):
    """Launches under TV_ATTN_STABLE_INPUTS behind the mask kernel, without a synchronisation: the one buffer of lengths, node
    counts (and pages) is rewritten in front of every mask call.  Each gives the bits it gives alone."""
    cfg = CONFIGS[0].scaled(B=B, L=1, Hq=G * Hkv, Hkv=Hkv, d=64, S_lo=1, S_hi=1000, Scap=1024, N=20, D=6, V=0, tree="uniform")
    c = make_case(cfg, seed=B, device="cuda", with_logits=False)
    N, d, steps = cfg.N, cfg.d, 10
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    if paged:
        kp, vp = (c[k].reshape(1, B, Hkv, 8, 128, d).transpose(2, 3).reshape(1, B * 8, Hkv, 128, d).contiguous() for k in ("k_cache", "v_cache"))
        tables = [torch.randperm(B * 8, device="cuda", generator=g).to(torch.int32).view(B, 8) for _ in range(steps)]
        table = torch.zeros_like(tables[0])
    lengths = [torch.randint(0, 1025, (B,), dtype=torch.int32, device="cuda", generator=g) for _ in range(steps)]
    counts = [torch.randint(1, N + 1, (B,), dtype=torch.int32, device="cuda", generator=g) for _ in range(steps)]
    S, n = torch.zeros_like(lengths[0]), torch.ones_like(counts[0])
    bits = torch.zeros(B, N, 1, dtype=torch.int32, device="cuda")
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    ws = torch.zeros(tv.tv_attn_workspace_bytes(B, N, cfg.Hq, Hkv, d, 1024), dtype=torch.uint8, device="cuda")

    def steps_with(sync):
        outs = [torch.zeros(1, B, N, cfg.Hq, d, dtype=torch.bfloat16, device="cuda") for _ in range(steps)]
        torch.cuda.synchronize()
        for s in range(steps):
            if paged:
                table.copy_(tables[s])
            S.copy_(lengths[s])
            torch.add(counts[s], 0, out=n)
            sync()
            tv.tree_build_mask(c["parent"], n, N - 1, 1, bits, status)
            sync()
            if paged:
                tv.tree_verify_attn_paged_layers(c["q"], kp, vp, table, c["k_tree"], c["v_tree"], S, n, bits, d ** -0.5, outs[s],
                                                 ws, status, flags=tv.TV_ATTN_STABLE_INPUTS)
            else:
                tv.tree_verify_attn_layers(c["q"], c["k_cache"], c["v_cache"], c["k_tree"], c["v_tree"], S, n, bits, d ** -0.5,
                                           outs[s], ws, status, flags=tv.TV_ATTN_STABLE_INPUTS)
            sync()
        torch.cuda.synchronize()
        return outs

    alone, behind = steps_with(torch.cuda.synchronize), steps_with(lambda: None)
    for s in range(steps):
        assert torch.equal(alone[s], behind[s]), s
    assert (i32(status) == 0).all()

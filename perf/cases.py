"""The measured work of this framework: verification steps of tree speculative decoding, as a serving program issues
them through the public entry points of ``paper_2603_08088_b200``.

A case names the shape of a step and how the program drives it:

  kind    "step"   mask, attention of L layers, acceptance, commit, on device buffers
          "split"  one member of a context-split group: attention over its share of the prefix, merge of all partials
          "host"   the whole step from pinned host buffers (``tv_verify_step_host``)
  calls   "fused" all layers in one call (``verify_step`` where the layout has it), "layer" one attention call per
          layer, as a teacher issues them whose layer l + 1 needs the output of layer l
  layout  "contiguous" (tree K/V in buffers of their own), "in_cache" (behind the prefix), "paged" (128-row pages)
  accept  "greedy", "sample" (temperature > 0), "none" (attention alone, with its log-sum-exp)

Values: Q, K and V are N(0, 1), so that a scaled score has unit variance; the logits of a greedy teacher are N(0, 1) with
a planted path of geometric length (three accepted tokens on average); the logits of a sampling teacher carry nearly all
of their mass on a few entries per row, the drafted tokens among them.
"""
import math

import numpy as np
import torch

import paper_2603_08088_b200 as tv

ROUNDS = 32            # prefix lengths in hand: a commit advances the ones it is given, so every pass takes the next
PAGE = 128
TEMPERATURE = 0.8
BF16 = 2


def _case(name, kind="step", calls="fused", layout="contiguous", accept="greedy", R=1, **shape):
    return dict(name=name, kind=kind, calls=calls, layout=layout, accept=accept, R=R, **shape)


def listed():
    return [
        # the smallest call there is: a toy model, where only latency and launches count
        _case("tiny_step", B=1, L=1, Hq=4, Hkv=2, d=64, S_lo=128, S_hi=128, N=15, D=4, V=1024),
        # interactive decoding, one sequence, one layer at a time of a model without grouped heads
        _case("one_sequence_mha_layer", B=1, L=1, Hq=32, Hkv=32, d=128, S_lo=2048, S_hi=2048, N=60, D=6, V=32000),
        # a whole step of interactive decoding with a small budget: every layer waits for the one below it
        _case("one_sequence_32_layers", calls="layer", B=1, L=32, Hq=32, Hkv=8, d=128, S_lo=1392, S_hi=1392, N=17, D=10,
              V=128256),
        # batched serving, prefixes of very different lengths
        _case("ragged_batch_layer", B=8, L=1, Hq=32, Hkv=8, d=128, S_lo=1024, S_hi=8192, N=64, D=7, V=128256),
        # paged serving with a budget of 64 drafted nodes: with the root 65, just past a multiple of the row tile
        _case("paged_batch_budget_64", layout="paged", B=8, L=8, Hq=32, Hkv=8, d=128, S_lo=512, S_hi=4096, N=65, D=10,
              V=32000),
        # the largest budget, drafted K/V written straight behind the prefix and reordered in place
        _case("in_cache_largest_budget", layout="in_cache", B=4, L=4, Hq=32, Hkv=8, d=128, S_lo=1024, S_hi=4096, N=256,
              D=16, V=32000),
        # long documents, one layer
        _case("long_context_layer", accept="none", B=4, L=1, Hq=32, Hkv=8, d=128, S_lo=32768, S_hi=32768, N=128, D=8, V=0),
        # the largest: a whole step of a batched 32-layer teacher
        _case("full_step_32_layers", B=16, L=32, Hq=32, Hkv=8, d=128, S_lo=512, S_hi=4096, N=60, D=6, V=153600),
        # the same batch where the layers depend on each other
        _case("batch_dependent_layers", calls="layer", B=16, L=8, Hq=32, Hkv=8, d=128, S_lo=512, S_hi=4096, N=60, D=6,
              V=153600),
        # sampling instead of greedy decoding
        _case("sampled_step", accept="sample", B=16, L=1, Hq=32, Hkv=8, d=128, S_lo=512, S_hi=4096, N=60, D=6, V=153600),
        # one of eight members that share the prefixes of long documents
        _case("context_split_member", kind="split", accept="none", R=8, B=4, L=1, Hq=32, Hkv=8, d=128, S_lo=32768,
              S_hi=32768, N=128, D=8, V=0),
        # a small teacher (seven query heads per KV head, odd vocabulary) whose activations come from host memory
        _case("host_buffers_step", kind="host", B=2, L=8, Hq=14, Hkv=2, d=64, S_lo=256, S_hi=1024, N=49, D=7, V=32003),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _cost_s(case):
    w = work(case)
    return max(w["bytes"] / 6e12, w["flops"] / 1e15)


def _state_bytes(case):
    kv = 2 * case["L"] * case["B"] * case["Hkv"] * case["d"] * (_capacity(case) + case["N"]) * BF16
    rows = case["B"] * case["N"]
    return kv + 2 * (1 + case["R"]) * case["L"] * rows * case["Hq"] * case["d"] * BF16 + rows * case["V"] * BF16


def draw(rng):
    largest = max(_cost_s(c) for c in listed())
    while True:
        kind = rng.choice(["step"] * 8 + ["split", "host"])
        accept = {"split": "none", "host": "greedy"}.get(kind) or rng.choice(["greedy"] * 5 + ["sample", "none"])
        layout = rng.choice(["contiguous", "contiguous", "in_cache", "paged"]) if kind == "step" else "contiguous"
        calls = rng.choice(["fused", "layer"]) if kind == "step" else "fused"
        Hkv = rng.choice([1, 2, 4, 8, 8, 16, 32])
        G = rng.choice([g for g in (1, 2, 3, 4, 4, 6, 7, 8) if g * Hkv <= 64])
        N = _log_int(rng, 8, 256)
        S_hi = _log_int(rng, 64, 32768)
        V = _log_int(rng, 1024, 153600)
        if rng.random() < 0.75:
            V = -(-V // 64) * 64
        case = dict(kind=kind, calls=calls, layout=layout, accept=accept, R=rng.choice([2, 4, 8]) if kind == "split" else 1,
                    B=_log_int(rng, 1, 32), L=1 if kind == "split" else _log_int(rng, 1, 32), Hq=G * Hkv, Hkv=Hkv,
                    d=rng.choice([64, 128, 128, 128]), S_lo=max(1, S_hi // rng.choice([1, 1, 4, 8])), S_hi=S_hi, N=N,
                    D=min(N - 1, rng.randint(3, 16)), V=V if accept != "none" else 0)
        if case["B"] * case["L"] * case["N"] * case["Hq"] * case["d"] > 1 << 27 and kind == "host":
            continue
        if _cost_s(case) <= 0.6 * largest and _state_bytes(case) <= 20e9:
            return case


def _capacity(case):
    rows = case["S_hi"] // case["R"] + case["N"]
    return -(-rows // PAGE) * PAGE + PAGE


def work(case):
    """Every input read once, every output written once; multiplications and additions of the attention."""
    B, L, N, Hq, Hkv, d, V, R = (case[k] for k in ("B", "L", "N", "Hq", "Hkv", "d", "V", "R"))
    keys = (case["S_lo"] + case["S_hi"]) / 2 / R
    rows = B * N * Hq * d
    by = L * (2 * B * Hkv * d * (keys + N) + 2 * rows) * BF16              # K/V of prefix and tree, Q, output
    by += B * N * V * BF16 + B * N * (3 + -(-N // 32)) * 4                 # logits, tree arrays, mask words
    if case["accept"] != "none":
        by += L * 2 * B * Hkv * d * 4 * BF16                               # rows committed (about four per sequence)
    else:
        by += L * B * Hq * N * 4                                           # log-sum-exp
    if case["kind"] == "split":
        by += (R + 1) * rows * BF16 + (R + 1) * B * Hq * N * 4             # the merge
    return {"bytes": by, "flops": 4.0 * L * Hq * N * d * B * (keys + N)}


def tolerance(case):
    # bf16 outputs from P rounded to bf16.  Against the same attention in 64 bits (three units of every contiguous case) the
    # relative error is 2.2e-3 to 2.9e-3 (2-norm), the largest difference 1.4 % of the rms: about four times that.  Whole
    # numbers and committed bytes are exact.
    return {"rel": 1e-2, "max": 0.06}


# ------------------------------------------------------------------------------------------------ inputs
def _tree(N, D, rng):
    """Parents of a tree of depth D: a spine of D nodes (the drafter's best path), every other node below a uniformly
    chosen node that is less than D deep.  parent < child."""
    parent, depth = np.full(N, -1, np.int32), np.zeros(N, np.int32)
    for i in range(1, N):
        p = i - 1 if i <= D else int(rng.integers(0, i))
        while depth[p] >= D:
            p = int(rng.integers(0, i))
        parent[i], depth[i] = p, depth[p] + 1
    return parent


def _logits(case, parent, tokens, rng, gen, dev):
    B, N, V = case["B"], case["N"], case["V"]
    logits = torch.empty(B, N, V, dtype=torch.bfloat16, device=dev).normal_(generator=gen)
    b, n, t, x = [], [], [], []
    for s in range(B):
        length = min(case["D"], int(rng.geometric(0.25)))          # planted path: the first nodes of the spine
        for i in range(1, N):
            if case["accept"] == "sample":
                b.append(s), n.append(int(parent[s, i])), t.append(int(tokens[s, i])), x.append(rng.uniform(16, 18))
            elif i <= length:
                b.append(s), n.append(i - 1), t.append(int(tokens[s, i])), x.append(16.0)
    if case["accept"] == "sample":                                 # what the drafter did not propose
        for s in range(B):
            for i in range(N):
                for tok in rng.integers(0, V, 6):
                    b.append(s), n.append(i), t.append(int(tok)), x.append(rng.uniform(12, 15))
    at = [torch.tensor(v, dtype=torch.int64, device=dev) for v in (b, n, t)]
    logits.view(-1)[(at[0] * N + at[1]) * V + at[2]] = torch.tensor(x, dtype=torch.bfloat16, device=dev)
    return logits


def prepare(case, seed):
    dev = torch.device("cuda")
    B, L, N, Hq, Hkv, d, V, R = (case[k] for k in ("B", "L", "N", "Hq", "Hkv", "d", "V", "R"))
    D, Dp1, cap = case["D"], case["D"] + 1, _capacity(case)
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed * 7919 + 17)

    def normal(*shape):
        return torch.empty(shape, dtype=torch.bfloat16, device=dev).normal_(generator=gen)

    def ints(a):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(dev)

    parent = np.stack([_tree(N, D, rng) for _ in range(B)])
    tokens = rng.integers(0, max(V, 1024), (B, N)).astype(np.int32)
    strata = np.linspace(case["S_lo"], case["S_hi"] + 1, B + 1)    # prefix lengths spread over the range
    S = np.floor(strata[:-1] + rng.random(B) * (strata[1:] - strata[:-1])).astype(np.int32).clip(case["S_lo"], case["S_hi"])
    S = rng.permutation(S) // R
    start = ints(np.tile(S, (ROUNDS, 1)))
    rounds = start.clone()
    st = {"case": case, "turn": 0, "start": start, "rounds": rounds, "prefix": list(rounds), "scale": d ** -0.5}
    c = {"parent": ints(parent), "n_nodes": ints(np.full(B, N)), "tokens": ints(tokens), "prefix_len": st["prefix"][0],
         "q": normal(L, B, N, Hq, d), "k_tree": normal(L, B, N, Hkv, d), "v_tree": normal(L, B, N, Hkv, d)}
    if case["layout"] == "paged":
        blocks = cap // PAGE
        st["k_pages"], st["v_pages"] = normal(L, B * blocks, Hkv, PAGE, d), normal(L, B * blocks, Hkv, PAGE, d)
        st["table"] = ints(rng.permutation(B * blocks).reshape(B, blocks))
    else:
        c["k_cache"], c["v_cache"] = normal(L, B, Hkv, cap, d), normal(L, B, Hkv, cap, d)
    if V:
        c["logits"] = _logits(case, parent, tokens, rng, gen, dev)
    st["inputs"] = c
    if case["accept"] == "sample":
        st["u_node"] = torch.from_numpy(rng.random((B, N), dtype=np.float32)).to(dev)
        st["u_bonus"] = torch.from_numpy(rng.random(B, dtype=np.float32)).to(dev)
        st["sample_ws"] = torch.zeros(tv.tv_sample_workspace_bytes(B, N, V), dtype=torch.uint8, device=dev)
    if case["kind"] == "host":
        st["host"] = {k: c.pop(k).cpu().pin_memory() for k in ("parent", "n_nodes", "tokens", "q", "k_tree", "v_tree", "logits")}
        pinned = dict(dtype=torch.int32, pin_memory=True)
        st["host"].update(out=torch.zeros(L, B, N, Hq, d, dtype=torch.bfloat16, pin_memory=True),
                          accept_len=torch.zeros(B, **pinned), accepted_nodes=torch.zeros(B, Dp1, **pinned),
                          next_token=torch.zeros(B, **pinned), status=torch.zeros(B, **pinned), retrieve_indices=None, P=N)
        st["staging"] = torch.zeros(tv.tv_step_staging_bytes(L, B, N, Hq, Hkv, d, cap, V, N, Dp1), dtype=torch.uint8, device=dev)
        return st
    st["buf"] = tv.StepBuffers(L, B, N, Hq, Hkv, d, cap, V, N, Dp1, device=dev, want_lse=case["accept"] == "none")
    if case["kind"] == "split":        # the partials the other members have sent; this member is the last, with the tree
        st["o_parts"] = normal(R, B, N, Hq, d).mul_(0.05)
        st["lse_parts"] = torch.rand(R, B, Hq, N, generator=gen, device=dev) + (math.log(max(1, case["S_hi"] // R)) + 0.5)
        st["out"] = torch.zeros(B, N, Hq, d, dtype=torch.bfloat16, device=dev)
        st["lse"] = torch.zeros(B, Hq, N, dtype=torch.float32, device=dev)
    return st


# ------------------------------------------------------------------------------------------------ one pass
def _next_prefix(st):
    """The prefix lengths of this pass: the ones a commit has advanced are not used again."""
    k = st["turn"] % ROUNDS
    if k == 0 and st["turn"]:
        st["rounds"].copy_(st["start"])
    st["turn"] += 1
    return st["prefix"][k]


def _attention(st, c, buf, prefix):
    case = st["case"]
    in_cache = case["layout"] == "in_cache"
    kt, vt = (None, None) if in_cache else (c["k_tree"], c["v_tree"])
    if case["layout"] == "paged":
        if case["calls"] == "fused":
            tv.tree_verify_attn_paged_layers(c["q"], st["k_pages"], st["v_pages"], st["table"], kt, vt, prefix, c["n_nodes"],
                                             buf.anc_bits, st["scale"], buf.out, buf.attn_ws, buf.status, lse=buf.lse,
                                             flags=tv.TV_ATTN_STABLE_INPUTS)
            return
        for l in range(case["L"]):
            tv.tree_verify_attn_paged(c["q"][l], st["k_pages"][l], st["v_pages"][l], st["table"], kt[l], vt[l], prefix,
                                      c["n_nodes"], buf.anc_bits, st["scale"], buf.out[l], buf.attn_ws, buf.status,
                                      lse=None if buf.lse is None else buf.lse[l])
        return
    if case["calls"] == "fused":
        tv.tree_verify_attn_layers(c["q"], c["k_cache"], c["v_cache"], kt, vt, prefix, c["n_nodes"], buf.anc_bits, st["scale"],
                                   buf.out, buf.attn_ws, buf.status, lse=buf.lse, flags=tv.TV_ATTN_STABLE_INPUTS)
        return
    for l in range(case["L"]):
        tv.tree_verify_attn(c["q"][l], c["k_cache"][l], c["v_cache"][l], None if in_cache else kt[l],
                            None if in_cache else vt[l], prefix, c["n_nodes"], buf.anc_bits, st["scale"], buf.out[l],
                            buf.attn_ws, buf.status, lse=None if buf.lse is None else buf.lse[l])


def _commit(st, c, buf, prefix):
    if st["case"]["layout"] == "paged":
        tv.kv_commit_paged(st["k_pages"], st["v_pages"], st["table"], c["k_tree"], c["v_tree"], buf.accepted_nodes,
                           buf.accept_len, prefix, buf.status)
    elif st["case"]["layout"] == "in_cache":
        tv.kv_commit_inplace(c["k_cache"], c["v_cache"], buf.accepted_nodes, buf.accept_len, prefix, st["case"]["N"], buf.status)
    else:
        tv.kv_commit(c["k_cache"], c["v_cache"], c["k_tree"], c["v_tree"], buf.accepted_nodes, buf.accept_len, prefix, buf.status)


def run(state):
    st, case, c = state, state["case"], state["inputs"]
    prefix = _next_prefix(st)
    if case["kind"] == "host":
        tv.tv_verify_step_host(st["host"], c["k_cache"], c["v_cache"], prefix, st["staging"], st["scale"], case["V"])
        h = st["host"]
        return [h["out"], h["accept_len"], h["accepted_nodes"], h["next_token"], h["status"], c["k_cache"], c["v_cache"], prefix]
    buf = st["buf"]
    if case["kind"] == "split":
        tv.tree_build_mask(c["parent"], c["n_nodes"], case["D"], case["N"], buf.anc_bits, buf.status)
        last = case["R"] - 1
        tv.tree_verify_attn(c["q"][0], c["k_cache"][0], c["v_cache"][0], c["k_tree"][0], c["v_tree"][0], prefix, c["n_nodes"],
                            buf.anc_bits, st["scale"], st["o_parts"][last], buf.attn_ws, buf.status, lse=st["lse_parts"][last])
        tv.tree_merge_partials(st["o_parts"], st["lse_parts"], st["out"], st["lse"])
        return [st["o_parts"][last], st["lse_parts"][last], st["out"], st["lse"], buf.status]
    if case["accept"] == "greedy" and case["calls"] == "fused" and case["layout"] != "paged":
        c["prefix_len"] = prefix
        tv.verify_step(c, buf, st["scale"], in_cache=case["layout"] == "in_cache")
    else:
        tv.tree_build_mask(c["parent"], c["n_nodes"], case["D"], case["N"], buf.anc_bits, buf.status, depth=buf.depth,
                           anc_table=buf.anc_table, retrieve_indices=buf.retrieve, n_paths=buf.n_paths)
        _attention(st, c, buf, prefix)
        if case["accept"] == "greedy":
            tv.tree_accept(c["logits"], c["tokens"], buf.retrieve, c["n_nodes"], buf.argmax_tok, buf.accept_len, buf.best_path,
                           buf.accepted_nodes, buf.next_token, buf.accept_ws, buf.status)
        elif case["accept"] == "sample":
            tv.tree_accept_sample(c["logits"], c["tokens"], c["parent"], c["n_nodes"], st["u_node"], st["u_bonus"], TEMPERATURE,
                                  buf.accept_len, buf.accepted_nodes, buf.next_token, st["sample_ws"], buf.status)
        if case["accept"] != "none":
            _commit(st, c, buf, prefix)
    outs = [buf.out, buf.status, buf.anc_bits, buf.depth, buf.anc_table, buf.retrieve, buf.n_paths]
    if case["accept"] == "none":
        return outs + [buf.lse]
    outs += [buf.accept_len, buf.accepted_nodes, buf.next_token, prefix]
    if case["accept"] == "greedy":
        outs += [buf.argmax_tok, buf.best_path]
    caches = [st["k_pages"], st["v_pages"]] if case["layout"] == "paged" else [c["k_cache"], c["v_cache"]]
    return outs + caches

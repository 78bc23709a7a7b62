"""The failure path of tree_verify_attn: every wait inside the kernel is bounded, and when one expires the
launch must end by itself - all roles leave their loops, the tensor memory is freed, TV_ST_TIMEOUT is raised
for every sequence - and the device must go on working.  The expiry is produced the harmless way: a test
entry point (treeverify_debug.h) launches the kernel with a limit of two milliseconds and a producer warp
that issues no copy, so the wait of the MMA-issuing warp for its first operands runs out - or with pieces of
cut units that are never announced, so the bounded poll of the merging piece runs out.  Nothing traps, faults or
waits without limit."""
import numpy as np
import pytest
import torch

import paper_2603_08088_b200 as tv
from workloads import CONFIGS, make_case
from gpu_util import i32

pytestmark = pytest.mark.gpu

SHAPES = [
    ("one_row_tile", 0, dict(B=2, S_lo=100, S_hi=300, Scap=320, N=15)),
    ("two_row_tiles_cut_units", 4, dict(B=6, L=1, V=0)),
]


@pytest.mark.parametrize("name,ci,over", SHAPES, ids=[s[0] for s in SHAPES])
def test_expired_wait_ends_the_launch_with_a_status_and_the_next_launch_is_unharmed(name, ci, over):
    cfg = CONFIGS[ci].scaled(**over)
    d = make_case(cfg, seed=31 + ci, device="cuda", with_logits=False)
    B, N, Hq, Hkv, dh = cfg.B, cfg.N, cfg.Hq, cfg.Hkv, cfg.d
    bits = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(d["parent"], d["n_nodes"], N - 1, 1, bits, status)
    ws = torch.zeros(max(256, tv.tv_attn_workspace_bytes(B, N, Hq, Hkv, dh, cfg.Scap)), dtype=torch.uint8, device="cuda")
    args = (d["q"][0], d["k_cache"][0], d["v_cache"][0], d["k_tree"][0], d["v_tree"][0], d["prefix_len"], d["n_nodes"],
            bits, dh ** -0.5)

    def normal():
        out = torch.full((B, N, Hq, dh), 3.0, dtype=torch.bfloat16, device="cuda")
        lse = torch.full((B, Hq, N), 3.0, dtype=torch.float32, device="cuda")
        tv.tree_verify_attn(*args, out, ws, status, lse=lse)
        torch.cuda.synchronize()
        return out, lse

    before = normal()
    assert (i32(status) == 0).all()
    # mode 0 of the test entry point is an ordinary launch (short limit, nothing withheld): same bits, no flag
    out0 = torch.zeros_like(before[0])
    tv.tv_debug_attn_expire(*args, out0, ws, status, 500_000_000, 0)
    torch.cuda.synchronize()
    assert (i32(status) == 0).all() and torch.equal(out0, before[0])

    modes = [1, 1, 1] + ([2, 2] if ci == 4 else [])       # 2: the merger's poll (only the second shape has cut units)
    for rep, mode in enumerate(modes):
        junk = torch.zeros_like(before[0])
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        tv.tv_debug_attn_expire(*args, junk, ws, status, 2_000_000, mode)    # 2 ms; 1: producer issues nothing
        t1.record()
        torch.cuda.synchronize()                                             # the launch returned by itself
        assert (i32(status) & tv.TV_ST_TIMEOUT != 0).all(), f"status {i32(status).tolist()}"
        assert (i32(status) & ~tv.TV_ST_TIMEOUT == 0).all()
        ms = t0.elapsed_time(t1)
        assert 1.5 <= ms <= 200.0, f"the expiring launch took {ms} ms"
        status.zero_()
        after = normal()                                                     # tensor memory was freed, barriers are fresh
        assert (i32(status) == 0).all()
        assert torch.equal(after[0], before[0]) and torch.equal(after[1], before[1])


MIDDLE = [(128, 4, 64), (64, 4, 64), (128, 4, 20), (64, 4, 20)]      # d, G, nodes: two row tiles and one, both head widths


@pytest.mark.parametrize("d,G,N", MIDDLE)
def test_waits_that_expire_anywhere_in_the_tile_loop(d, G, N):
    """Limits of the order of the waits themselves: whichever wait is the first to be longer gives up, in the tile loop too,
    where the lanes of a softmax warp do so one by one with collective instructions behind the wait.  A launch either
    finishes or reports; the one behind it is unharmed."""
    cfg = CONFIGS[0].scaled(B=40, L=1, Hq=2 * G, Hkv=2, d=d, S_lo=2500, S_hi=3000, Scap=3200, N=N, D=6, V=0, tree="uniform")
    c = make_case(cfg, seed=d + N, device="cuda", with_logits=False)
    bits = torch.zeros(cfg.B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    status = torch.zeros(cfg.B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(c["parent"], c["n_nodes"], N - 1, 1, bits, status)
    ws = torch.zeros(tv.tv_attn_workspace_bytes(cfg.B, N, cfg.Hq, 2, d, cfg.Scap), dtype=torch.uint8, device="cuda")
    args = (c["q"][0], c["k_cache"][0], c["v_cache"][0], c["k_tree"][0], c["v_tree"][0], c["prefix_len"], c["n_nodes"], bits,
            d ** -0.5)
    before, after = (torch.full((cfg.B, N, cfg.Hq, d), x, dtype=torch.bfloat16, device="cuda") for x in (3.0, 4.0))
    tv.tree_verify_attn(*args, before, ws, status)
    torch.cuda.synchronize()
    assert (i32(status) == 0).all()
    expired = 0
    for limit in (0, 1000, 2000, 4000, 8000, 16000, 500_000_000):
        got = torch.zeros_like(before)
        tv.tv_debug_attn_expire(*args, got, ws, status, limit, 0)
        torch.cuda.synchronize()
        st = i32(status)
        assert (st == st[0]).all() and st[0] in (0, tv.TV_ST_TIMEOUT)
        assert st[0] != 0 or torch.equal(got, before)
        expired += st[0] != 0
        status.zero_()
        tv.tree_verify_attn(*args, after, ws, status)
        torch.cuda.synchronize()
        assert (i32(status) == 0).all() and torch.equal(before, after)
    assert expired >= 1


@pytest.mark.parametrize("N,d", [(65, 64), (129, 128)])
def test_waits_that_expire_in_two_launches_at_the_same_time(N, d):
    """The shapes whose odd last row tile has a launch beside the others, of one row tile per CTA: waits of either launch run out, in
    the tile loop, for operands that nobody sends and for pieces that are never announced.  Both end, the status says so, and the
    pair behind them on the same workspace gives its bits."""
    B, Hkv, G, cap = 14, 8, 4, 10240
    cfg = CONFIGS[0].scaled(B=B, L=1, Hq=G * Hkv, Hkv=Hkv, d=d, S_lo=2600, S_hi=4300, Scap=cap, N=N, D=6, V=0, tree="uniform")
    c = make_case(cfg, seed=d + N, device="cuda", with_logits=False)
    bits = torch.zeros(B, N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(c["parent"], c["n_nodes"], N - 1, 1, bits, status)
    ws = torch.zeros(tv.tv_attn_workspace_bytes(B, N, cfg.Hq, Hkv, d, cap), dtype=torch.uint8, device="cuda")
    args = (c["q"][0], c["k_cache"][0], c["v_cache"][0], c["k_tree"][0], c["v_tree"][0], c["prefix_len"], c["n_nodes"], bits, d ** -0.5)
    before, after = (torch.full((B, N, cfg.Hq, d), x, dtype=torch.bfloat16, device="cuda") for x in (3.0, 4.0))
    n0 = tv.tv_launch_count()
    tv.tree_verify_attn(*args, before, ws, status)
    assert tv.tv_launch_count() - n0 == 2
    torch.cuda.synchronize()
    assert (i32(status) == 0).all()
    for limit, mode in [(x, 0) for x in (0, 1000, 2000, 4000, 8000, 16000, 500_000_000)] + [(2_000_000, 1), (2_000_000, 2), (2_000_000, 33)]:
        got = torch.zeros_like(before)
        tv.tv_debug_attn_expire(*args, got, ws, status, limit, mode)
        torch.cuda.synchronize()
        st = i32(status)
        assert (st == st[0]).all() and st[0] in ((0, tv.TV_ST_TIMEOUT) if mode == 0 else (tv.TV_ST_TIMEOUT,)), (limit, mode)
        assert st[0] != 0 or torch.equal(got, before)
        status.zero_()
        tv.tree_verify_attn(*args, after, ws, status)
        torch.cuda.synchronize()
        assert (i32(status) == 0).all() and torch.equal(before, after), (limit, mode)


def test_expired_waits_of_the_cluster_kernel():
    """As above, with a producer that issues nothing: every CTA of a cluster gives up, meets the others at the cluster's barriers
    and leaves."""
    cfg = CONFIGS[0].scaled(B=1, L=1, Hq=8, Hkv=2, d=128, S_lo=900, S_hi=900, Scap=1000, N=40, D=6, V=0, tree="uniform")
    c = make_case(cfg, seed=3, device="cuda", with_logits=False)
    bits = torch.zeros(1, 40, 2, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    tv.tree_build_mask(c["parent"], c["n_nodes"], 39, 1, bits, status)
    ws = torch.zeros(tv.tv_attn_workspace_bytes(1, 40, 8, 2, 128, 1000), dtype=torch.uint8, device="cuda")
    args = (c["q"][0], c["k_cache"][0], c["v_cache"][0], c["k_tree"][0], c["v_tree"][0], c["prefix_len"], c["n_nodes"], bits, 0.1)
    before, got = torch.zeros(1, 40, 8, 128, dtype=torch.bfloat16, device="cuda"), torch.zeros(1, 40, 8, 128, dtype=torch.bfloat16, device="cuda")
    tv.tree_verify_attn(*args, before, ws, status)
    tv.tv_debug_attn_expire(*args, got, ws, status, 500_000_000, 16)
    torch.cuda.synchronize()
    assert (i32(status) == 0).all() and torch.equal(before, got)          # the same kernel, bit for bit
    for _ in range(3):
        tv.tv_debug_attn_expire(*args, got, ws, status, 2_000_000, 17)
        torch.cuda.synchronize()
        assert i32(status).tolist() == [tv.TV_ST_TIMEOUT]
        status.zero_()
        tv.tree_verify_attn(*args, got, ws, status)
        torch.cuda.synchronize()
        assert (i32(status) == 0).all() and torch.equal(before, got)

"""Device-side guards: what the kernels do with data they cannot trust.

The copy kernels turn device-resident integers (kept indices, block-table entries, tree-path
nodes, sequence lengths) into addresses.  Each guard is fed one value that is outside the range
the call's arguments declare but still inside the tensor the test allocated, so that no access
could leave the allocation even if a guard were missing.  Expected: the offending row is skipped
(its destination keeps the sentinel it held), every other row equals the oracle, and
SPECVLM_ERR_INVALID_ARG arrives in d_status.  One test makes a bounded barrier wait run out
on a barrier nothing arrives at and reads SPECVLM_ERR_TIMEOUT back; the kernel returns normally.
The last one checks what attention makes of the partial results of a CTA that gave up."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from gpu_util import host_view, make_cache
from helpers import bits
from paper_2508_16201_b200 import specvlm, synth

pytestmark = pytest.mark.gpu


def _status():
    return torch.zeros(1, dtype=torch.int32, device="cuda")


def _shrunk(cache, n_blocks):
    """The same memory described as a cache of only n_blocks physical blocks."""
    return specvlm.KvCache(cache.k[:, :n_blocks], cache.v[:, :n_blocks], cache.seq_lens, cache.max_seq_len,
                           cache.block_table)


@pytest.mark.parametrize("bad", [-1, "video_len+2"])
def test_gather_skips_kept_index_outside_the_video(bad):
    L, H, D = 2, 2, 128
    vs, nv, nt = 4, 392, 40                       # 4 prefix tokens, so index -1 is still inside the tensor
    src_len = vs + nv + nt
    rng = np.random.default_rng(1)
    kept = np.sort(rng.choice(nv, 39, replace=False)).astype(np.int32)
    src, sk, sv = make_cache(L, H, D, [src_len], paged=False, seed=70)
    dst_len = src_len - nv + len(kept)
    dst, _, _ = make_cache(L, H, D, [dst_len], paged=False, seed=71)
    before = host_view(dst.k, None, [dst_len])[0].copy()
    corrupt = kept.copy()
    corrupt[17] = -1 if bad == -1 else nv + 2
    st = _status()
    specvlm.gather_kv(src, torch.from_numpy(corrupt).cuda(), [0, len(kept)], [vs], [nv], [src_len], dst, d_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == specvlm.ERR_INVALID_ARG
    ref = oracle.gather_kv(sk[0], kept, vs, nv, src_len)
    got = host_view(dst.k, None, [dst_len])[0]
    j = vs + 17                                   # destination position of the corrupted entry
    keep = np.ones(dst_len, dtype=bool)
    keep[j] = False
    assert np.array_equal(got[:, :, keep], ref[:, :, keep])
    assert np.array_equal(got[:, :, j], before[:, :, j])          # skipped: nothing written there


@pytest.mark.parametrize("side", ["src", "dst"])
def test_gather_skips_block_outside_the_declared_pool(side):
    L, H, D = 1, 2, 64
    nv, nt = 196, 60
    src_len = nv + nt
    kept = np.arange(0, nv, 10, dtype=np.int32)
    dst_len = nt + len(kept)
    src, sk, _ = make_cache(L, H, D, [src_len], paged=True, seed=72)
    dst, _, _ = make_cache(L, H, D, [dst_len], paged=True, seed=73)
    st = _status()
    c = src if side == "src" else dst
    top = int(c.block_table.max())                # the highest physical block in use ...
    small = _shrunk(c, top)                       # ... is outside a pool declared one block shorter
    before = host_view(dst.k, dst.block_table, [dst_len])[0].copy()
    specvlm.gather_kv(small if side == "src" else src, torch.from_numpy(kept).cuda(), [0, len(kept)], [0], [nv],
                      [src_len], small if side == "dst" else dst, d_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == specvlm.ERR_INVALID_ARG
    ref = oracle.gather_kv(sk[0], kept, 0, nv, src_len)
    got = host_view(dst.k, dst.block_table, [dst_len])[0]
    table = c.block_table.cpu().numpy()[0]
    lb = int(np.where(table == top)[0][0])        # logical block that maps to the refused one
    if side == "dst":
        bad_rows = np.arange(dst_len) // 64 == lb
    else:
        src_pos = np.concatenate([kept, np.arange(nv, src_len)])
        bad_rows = src_pos // 64 == lb
    assert bad_rows.any() and not bad_rows.all()
    assert np.array_equal(got[:, :, ~bad_rows], ref[:, :, ~bad_rows])
    assert np.array_equal(got[:, :, bad_rows], before[:, :, bad_rows])


def test_append_overflowing_sequence_writes_no_row_at_all():
    L, H, D, n_new = 2, 2, 64, 4
    cache, k_host, v_host = make_cache(L, H, D, [20, 20], paged=False, seed=74, extra_capacity=8)
    cache.seq_lens.copy_(torch.tensor([18, 10], dtype=torch.int32))     # 18 + 4 > 20: two rows would still fit
    new = synth.randn_bf16((L, 2, n_new, H, D), "cuda", 75, "n")
    st = _status()
    specvlm.append_kv(cache, new, new, d_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == specvlm.ERR_INVALID_ARG
    assert cache.seq_lens.cpu().tolist() == [18, 14]
    got = host_view(cache.k, None, [20, 20])
    assert np.array_equal(got[0], k_host[0])                              # rows 18, 19 included
    rk, n = oracle.append_kv(k_host[1][:, :, :14].copy(), bits(new[:, 1]), 10)
    assert n == 14 and np.array_equal(got[1][:, :, :14], rk[:, :, :14])


def test_append_skips_block_outside_the_declared_pool():
    L, H, D, n_new = 1, 2, 64, 3
    lens = [62]                                   # the new rows 62, 63 | 64 straddle two pages
    cache, k_host, _ = make_cache(L, H, D, [lens[0] + n_new], paged=True, seed=76)
    cache.seq_lens.copy_(torch.tensor(lens, dtype=torch.int32))
    table = cache.block_table.cpu().numpy()[0]
    second = int(table[1])
    if second < int(table[0]):                    # make the second page the one outside the pool
        pytest.skip("page order of this seed puts the first page last")
    small = _shrunk(cache, second)
    new = synth.randn_bf16((L, 1, n_new, H, D), "cuda", 77, "n")
    st = _status()
    specvlm.append_kv(small, new, new, d_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == specvlm.ERR_INVALID_ARG
    got = host_view(cache.k, cache.block_table, [lens[0] + n_new])[0]
    nb = bits(new[:, 0])                          # [L][n_new][H][D]
    assert np.array_equal(got[:, :, 62], nb[:, 0]) and np.array_equal(got[:, :, 63], nb[:, 1])
    assert np.array_equal(got[:, :, 64], k_host[0][:, :, 64])             # the refused page is untouched


@pytest.mark.parametrize("bad_node", [0, "n_nodes"])
def test_compact_tree_skips_path_node_outside_the_window(bad_node):
    L, H, D, n_nodes = 2, 2, 128, 8
    old = 100
    cache, k_host, _ = make_cache(L, H, D, [old + n_nodes], paged=False, seed=78, extra_capacity=16)
    path_ok = [2, 5, 7] + [-1] * (n_nodes - 3)
    path = list(path_ok)
    path[1] = 0 if bad_node == 0 else n_nodes     # position old + n_nodes is inside the spare capacity
    st = _status()
    acc = torch.tensor([3], dtype=torch.int32, device="cuda")
    specvlm.compact_tree_kv(cache, torch.tensor([path], dtype=torch.int32, device="cuda"), acc, d_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == specvlm.ERR_INVALID_ARG
    ref, n = oracle.compact_tree_kv(k_host[0].copy(), old + n_nodes, n_nodes, path_ok[:3])
    assert int(cache.seq_lens[0]) == n
    got = host_view(cache.k, None, [old + n_nodes])[0]
    rows = np.ones(old + n_nodes, dtype=bool)
    rows[old + 2] = False                         # the destination of the refused move
    rows[n:] = False                              # past the new end nothing is specified
    assert np.array_equal(got[:, :, rows], ref[:, :, rows])
    assert np.array_equal(got[:, :, old + 2], k_host[0][:, :, old + 2])


def test_bounded_wait_runs_out_and_reports_timeout():
    st = _status()
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    specvlm.debug_wait_timeout(5, st, flag)
    t1.record()
    torch.cuda.synchronize()                      # returns: the kernel gave up by itself
    assert int(st.item()) == specvlm.ERR_TIMEOUT and int(flag.item()) == 1
    assert "timed out" in specvlm.status_string(int(st.item()))
    ms = t0.elapsed_time(t1)
    assert 4.0 <= ms <= 500.0, ms
    # the context is intact: an ordinary call still works afterwards
    logits, drafts = synth.logits_and_drafts(1, 2, 1024, "cuda", 9)
    n, nxt, _ = specvlm.accept(logits, drafts)
    a, nx, _ = oracle.accept(logits[0].cpu().numpy(), drafts[0].cpu().numpy())
    assert (int(n[0]), int(nxt[0])) == (a, nx)


@pytest.mark.parametrize("Hq,Hkv,gamma,D,lens", [
    (28, 4, 0, 128, [6000]),                     # 16-row slices, few items in many parts (four warps share the parts)
    (28, 4, 0, 64, [700, 0, 3000, 129] * 3),     # the same with items that no boundary cuts and empty sequences
    (64, 8, 5, 128, [1500, 300]),                # 48 rows
    (16, 2, 8, 64, [3000, 300]),                 # 72 rows, d = 64
    (64, 4, 8, 128, [1100, 0, 2000]),            # 144 rows: two parts of the window per CTA
    (32, 2, 8, 64, [260, 2500])])                # the same at d = 64
def test_items_with_a_part_that_was_given_up_are_left_alone(Hq, Hkv, gamma, D, lens):
    """An item that slice boundaries cut is folded from several CTAs' partial results.  Where one of the CTAs gave
    up, nothing may be made of what its slots hold.  The second kernel of a finished call runs again over the call's
    scratch: as it is, it stores the cut items once more, bit for bit; with a CTA marked as having given up, all of them
    but the ones that this CTA has a part of, which keep a sentinel.  (No wait is made to expire.)"""
    L, B, nq = 2, len(lens), gamma + 1
    group, n_parts, q_per = Hq // Hkv, ctypes.c_int32(), ctypes.c_int32()
    assert specvlm.lib().specvlm_debug_window_parts(nq, group, ctypes.byref(n_parts), ctypes.byref(q_per)) == 0
    q_per = q_per.value                              # query tokens of a part of a window wider than 128 rows
    cache, _, _ = make_cache(L, Hkv, D, [max(n, 1) for n in lens], paged=False, seed=80)
    cache.seq_lens.copy_(torch.tensor(lens, dtype=torch.int32))
    q = synth.randn_bf16((L, B, nq, Hq, D), "cuda", 81, "Q")
    lse = torch.empty((L, B, nq, Hq), dtype=torch.float32, device="cuda")
    specvlm.debug_set_attn_splits(6 if gamma == 0 else 0)
    try:
        ws = torch.full((specvlm.attn_workspace_bytes(cache, B, Hq, gamma),), 255, dtype=torch.uint8, device="cuda")
        whole = specvlm.verify_attn(cache, q, gamma, 0.1, lse=lse, ws=ws)
        saved = ws.clone()

        def merge(cta=-1):
            """Items [part of the window][L][B][Hkv] that the merge has stored: whole, and as in the call."""
            out, lse2 = torch.full_like(whole, 7.0), torch.full_like(lse, 7.0)
            ws.copy_(saved)
            n = specvlm.debug_attn_merge(cache, out, ws, lse2, cta)
            stored = (out != 7.0).any(-1)
            assert torch.equal(stored, lse2 != 7.0)
            assert torch.equal(out[stored], whole[stored]) and torch.equal(lse2[stored], lse[stored])
            items = [h.unflatten(3, (Hkv, group)).transpose(2, 3).flatten(3) for h in stored.split(q_per, dim=2)]
            assert all(torch.equal(i.any(-1), i.all(-1)) for i in items)
            return n, torch.stack([i.all(-1) for i in items])

        n, cut = merge()
        assert cut.any()
        left, parts = torch.zeros_like(cut), 0
        for cta in range(n):
            stored = merge(cta)[1]
            assert not (stored & ~cut).any()
            left |= cut & ~stored
            parts += int((cut & ~stored).sum())
        assert torch.equal(left, cut) and parts >= 2 * int(cut.sum())   # a cut item has parts in two CTAs at least
    finally:
        specvlm.debug_set_attn_splits(0)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("splits,lens", [(0, [1500, 700, 0, 100]),       # a cluster per item; two of them left to one CTA
                                         (1, [1500, 40, 0, 300]),        # a CTA per item
                                         (5, [1500, 40, 0, 900])])       # slices
def test_decode_reports_a_cta_that_gives_up(splits, lens, paged, D):
    """Every CTA in turn gives up as if a wait of its had expired: the call reports it if the CTA had work, stores nothing for
    the items it has a part of (one item, or those of its slice), and everything else bit for bit.  No wait is made to
    expire."""
    L, Hkv, Hq, B = 1, 2, 8, len(lens)
    cache, _, _ = make_cache(L, Hkv, D, [max(n, 1) for n in lens], paged=paged, seed=82)
    cache.seq_lens.copy_(torch.tensor(lens, dtype=torch.int32))
    q = synth.randn_bf16((L, B, Hq, D), "cuda", 83, "Q")
    specvlm.debug_set_attn_splits(splits)
    try:
        ws = torch.full((specvlm.attn_workspace_bytes(cache, B, Hq, 0),), 255, dtype=torch.uint8, device="cuda")

        def run(cta):
            out, lse, st = torch.full_like(q, 7.0), torch.full((L, B, Hq), 7.0, device="cuda"), _status()
            n = specvlm.debug_attn_give_up(cache, q, 0.1, out, lse, ws, st, cta)
            torch.cuda.synchronize()
            return n, out, lse, int(st.item())

        n, whole, whole_lse, st = run(-1)
        assert st == 0 and torch.equal(whole, specvlm.draft_decode_attn(cache, q, 0.1, ws=ws)) and (whole_lse != 7.0).all()
        lost = torch.zeros((B, Hkv), dtype=torch.int32)
        for cta in range(n):
            _, out, lse, st = run(cta)
            stored = (out != 7.0).any(-1)
            assert torch.equal(stored, lse != 7.0)
            assert torch.equal(out[stored], whole[stored]) and torch.equal(lse[stored], whole_lse[stored])
            items = stored.view(B, Hkv, Hq // Hkv)
            assert torch.equal(items.any(-1), items.all(-1))
            left = ~items.all(-1)
            assert st == (specvlm.ERR_TIMEOUT if left.any() else 0)
            assert left.any() or splits != 1 or lens[cta // Hkv] == 0           # a CTA per item: all but the empty sequence's
            lost += left.cpu()
        for b, length in enumerate(lens):
            tiles = -(-length // 64)
            parts = min(tiles, 1 if splits == 1 or (splits == 0 and tiles <= 4) else 2)
            assert (lost[b] >= parts).all() and (parts > 1 or (lost[b] == parts).all()), (b, lost[b])
    finally:
        specvlm.debug_set_attn_splits(0)

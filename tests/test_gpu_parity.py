"""GPU parity: every C-ABI call against the CPU checker on the same seeded inputs.

Integer outputs (argmax ids, accepted path, next token, status, context lengths) and the committed
cache bytes must match exactly; the attention output must be within max-abs 2e-2 and max-rel 1e-2
of the checker's float64 result."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest
import torch

from paper_2408_00264_b200 import workloads as W
from parity_util import ATTN_MAX_REL, assert_attn_close, attn_errors, log_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def clv():
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA device")
    from paper_2408_00264_b200 import binding
    binding.lib()          # raises if the library was not built: there is no fallback
    return binding


def make_step(w, **kw):
    from paper_2408_00264_b200.step import VerifyStep
    return VerifyStep(w, **kw)


def bits(t):
    from paper_2408_00264_b200.step import bits_of
    return bits_of(t)


def check_attention(oracle, w, st, rows=None):
    if rows is None:
        ref, _, lse, status = oracle.tree_attn(w.q, w.k_cache, w.v_cache, w.k_tree, w.v_tree,
                                               w.parent, w.ctx_len, w.scale,
                                               block_table=w.block_table)
        got = bits(st.out)
        got_lse = st.lse.cpu().numpy().astype(np.float64)
    else:
        ref, _, lse, status = oracle.tree_attn(w.q, w.k_cache, w.v_cache, w.k_tree, w.v_tree,
                                               w.parent, w.ctx_len, w.scale,
                                               block_table=w.block_table, rows=rows)
        g = bits(st.out)
        got = g[rows[:, 0], rows[:, 1], rows[:, 2]]
        got_lse = st.lse.cpu().numpy().astype(np.float64)[rows[:, 0], rows[:, 1], rows[:, 2]]
    assert np.array_equal(st.status[0].cpu().numpy(), status)
    assert_attn_close(got, ref, w.cfg.name)
    assert np.abs(got_lse - lse).max() < 2e-3
    if w.cfg.name in W.CONFIGS:
        a, r = attn_errors(got, ref)
        log_parity(w.cfg.name, rows=int(np.prod(got.shape[:-1])), max_abs=a, max_row_rel=r,
                   max_lse_abs=float(np.abs(got_lse - lse).max()))
    return ref


def check_attention_status(oracle, w, st):
    """The checker's attention output in float64, after a look at the per-sequence status."""
    ref, _, _, status = oracle.tree_attn(w.q, w.k_cache, w.v_cache, w.k_tree, w.v_tree, w.parent, w.ctx_len, w.scale,
                                         block_table=w.block_table)
    assert np.array_equal(st.status[0].cpu().numpy(), status)
    return ref


def check_accept_and_commit(oracle, w, st):
    ids = oracle.argmax(w.logits, w.cfg.vocab)
    assert np.array_equal(st.ids.cpu().numpy(), ids)
    alen, aidx, nxt, s1 = oracle.accept_walk(w.parent, w.tokens, ids, w.path_cap)
    assert np.array_equal(st.accept_len.cpu().numpy(), alen)
    assert np.array_equal(st.accept_idx.cpu().numpy(), aidx)
    assert np.array_equal(st.next_token.cpu().numpy(), nxt)
    assert np.array_equal(st.status[1].cpu().numpy(), s1)
    kc, vc, new_len, s2 = oracle.kv_commit(w.k_cache, w.v_cache, w.k_tree, w.v_tree, aidx, alen,
                                           w.ctx_len, block_table=w.block_table)
    assert np.array_equal(st.ctx_len_out.cpu().numpy(), new_len)
    assert np.array_equal(st.status[2].cpu().numpy(), s2)
    assert np.array_equal(bits(st.k_cache), kc)      # whole buffers, byte for byte
    assert np.array_equal(bits(st.v_cache), vc)
    return alen


def full_step(clv, oracle, w, rows=None):
    st = make_step(w)
    st.run()
    torch.cuda.synchronize()
    check_attention(oracle, w, st, rows)
    alen = check_accept_and_commit(oracle, w, st)
    # a second step on fresh buffers gives bit-identical outputs (no stale workspace state)
    st2 = make_step(w)
    st2.workspace = st.workspace
    st2.run(fused_tail=False)   # the walk and the commit as two launches: same results as the fused one
    torch.cuda.synchronize()
    assert torch.equal(st2.ids, st.ids) and torch.equal(st2.accept_idx, st.accept_idx)
    assert torch.equal(st2.accept_len, st.accept_len) and torch.equal(st2.next_token, st.next_token)
    assert torch.equal(st2.ctx_len_out, st.ctx_len_out) and torch.equal(st2.status, st.status)
    assert torch.equal(st2.k_cache, st.k_cache) and torch.equal(st2.v_cache, st.v_cache)
    assert_attn_close(bits(st2.out), W.bf16_bits_to_f64(bits(st.out)), "repeat")
    return alen


# ------------------------------------------------------------------ the five stated workloads
@pytest.mark.parametrize("name", ["C1", "C2", "C3", "C4", "C5"])
def test_config_full_compare(clv, oracle, name):
    # every attention row, every id, the accepted paths and the whole committed cache, at the
    # stated sizes (the checker needs a few seconds for C4 and some tens of seconds for C5)
    w = W.generate(W.CONFIGS[name])
    alen = full_step(clv, oracle, w)
    assert (alen >= 1).all()


# ------------------------------------------------------------------ shapes around tile edges
@pytest.mark.parametrize("ctx", [0, 1, 63, 64, 65, 127, 129, 700])
@pytest.mark.parametrize("n_nodes,hq,hkv", [(1, 4, 4), (7, 4, 1), (33, 8, 2), (64, 4, 4),
                                            (128, 8, 2), (100, 6, 3)])
def test_attention_shapes(clv, oracle, ctx, n_nodes, hq, hkv):
    cfg = W.small_config(batch=2, n_q_heads=hq, n_kv_heads=hkv, ctx=ctx, n_nodes=n_nodes,
                         max_depth=6, vocab=64, seed=W.BASE_SEED + ctx * 131 + n_nodes)
    w = W.generate(cfg)
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st)


@pytest.mark.parametrize("tree", ["chain", "star", "forest"])
@pytest.mark.parametrize("paged", [False, True])
def test_attention_special_trees_and_paging(clv, oracle, tree, paged):
    n = 40
    cfg = W.small_config(batch=3, n_q_heads=8, n_kv_heads=2, ctx=(1, 300), n_nodes=n, vocab=64,
                         paged=paged)
    w = W.generate(cfg)
    w.parent[:] = {"chain": W.tree_chain, "star": W.tree_star, "forest": W.tree_forest}[tree](n)
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st)


@pytest.mark.parametrize("hq,hkv,n_nodes", [(6, 2, 37), (12, 2, 37), (5, 1, 37), (28, 4, 64), (24, 2, 128),
                                             (7, 1, 18), (7, 1, 19)])
def test_attention_group_sizes_that_do_not_divide_128(clv, oracle, hq, hkv, n_nodes):
    # a 128-row tile holds whole nodes only, so with such group sizes some of its rows stay idle
    cfg = W.small_config(batch=2, n_q_heads=hq, n_kv_heads=hkv, ctx=(30, 500), n_nodes=n_nodes, vocab=64,
                         seed=W.BASE_SEED + hq)
    w = W.generate(cfg)
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st)


def test_attention_many_splits_and_ragged(clv, oracle):
    # few (sequence, head) units and a long context: the key axis is split many ways; one
    # sequence is much shorter than max_ctx_len so some splits of it are empty
    cfg = W.small_config(batch=2, n_q_heads=2, n_kv_heads=1, ctx=(40, 2500), n_nodes=20, vocab=64,
                         seed=W.BASE_SEED + 9)
    w = W.generate(cfg)
    w.ctx_len[0] = 40
    st = make_step(w)
    st.max_ctx_len = 2500
    st.workspace = clv.new_workspace(st.shape, st.cache, 2500)
    st.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st)


def _scale_bf16_by_pow2(bits_arr, k):
    """bf16 bit patterns times 2^k, exactly (normal numbers; zeros stay zeros)."""
    b = bits_arr.astype(np.int64)
    expo = (b >> 7) & 0xFF
    new = np.clip(expo + k, 1, 254)
    out = (b & ~(0xFF << 7)) | (new << 7)
    return np.where(expo == 0, b, out).astype(np.uint16)


@pytest.mark.parametrize("k_lo,k_hi", [(40, 40), (-40, -40), (30, -30), (-30, 30)])
def test_attention_value_magnitudes_across_splits(clv, oracle, k_lo, k_hi):
    # The split-KV partial sums travel between blocks in fp16, every row scaled by its own power of
    # two.  Values far outside the fp16 range, and key ranges whose values differ by 2^60, must
    # come out as the checker computes them (relative to each output row's scale: the absolute
    # tolerance presupposes values of order one and is not applied here).
    from parity_util import attn_errors, ATTN_MAX_REL
    cfg = W.small_config(batch=2, n_q_heads=8, n_kv_heads=2, ctx=(1500, 2300), n_nodes=48, vocab=64,
                         seed=W.BASE_SEED + 77)
    w = W.generate(cfg)
    half = w.v_cache.shape[1] // 2 if w.v_cache.ndim == 4 else None
    assert half is not None
    w.v_cache[:, :half] = _scale_bf16_by_pow2(w.v_cache[:, :half], k_lo)
    w.v_cache[:, half:] = _scale_bf16_by_pow2(w.v_cache[:, half:], k_hi)
    w.v_tree[:] = _scale_bf16_by_pow2(w.v_tree, k_hi)
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    ref, _, lse, status = oracle.tree_attn(w.q, w.k_cache, w.v_cache, w.k_tree, w.v_tree, w.parent,
                                           w.ctx_len, w.scale, block_table=w.block_table)
    got = bits(st.out)
    assert np.array_equal(st.status[0].cpu().numpy(), status)
    assert np.isfinite(W.bf16_bits_to_f64(got)).all()
    _, rel = attn_errors(got, ref)
    assert rel <= ATTN_MAX_REL, rel
    assert np.abs(st.lse.cpu().numpy().astype(np.float64) - lse).max() < 2e-3


def test_attention_mask_exactness_on_device(clv, oracle):
    # overwriting K/V of nodes that are not ancestors must not change a node's output at all
    cfg = W.small_config(batch=1, n_q_heads=4, n_kv_heads=2, ctx=100, n_nodes=24, vocab=64)
    w = W.generate(cfg)
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    base = st.out.clone()
    i = 17
    anc = set()
    j = i
    while j >= 0:
        anc.add(j)
        j = int(w.parent[0, j])
    big = W.f32_to_bf16_bits(np.full(128, 3.0e4, np.float32))
    for j in range(24):
        if j not in anc:
            w.k_tree[0, j, :] = big
            w.v_tree[0, j, :] = big
    st2 = make_step(w)
    st2.tree_attn()
    torch.cuda.synchronize()
    assert torch.equal(st2.out[0, i], base[0, i])


def test_attention_flags_bad_sequences(clv, oracle):
    cfg = W.small_config(batch=3, n_q_heads=4, n_kv_heads=2, ctx=70, n_nodes=10, vocab=64)
    w = W.generate(cfg)
    w.parent[1, 4] = 6                      # parent after child
    st = make_step(w)
    st.ctx_len[2] = w.cap_tokens + 5        # context larger than the cache rows
    st.tree_attn()
    torch.cuda.synchronize()
    assert st.status[0].cpu().tolist() == [0, clv.CLV_ERR_TREE, clv.CLV_ERR_TREE]
    ref = oracle.tree_attn(w.q, w.k_cache, w.v_cache, w.k_tree, w.v_tree, w.parent, w.ctx_len,
                           w.scale)[0]
    assert_attn_close(bits(st.out)[0], ref[0], "valid sequence beside bad ones")


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("hq,hkv,n_nodes", [(4, 4, 16), (4, 4, 50), (8, 2, 32), (8, 2, 128)])
def test_attention_flags_the_largest_lengths_there_are(clv, oracle, hq, hkv, n_nodes, paged):
    # The number of a length's pages is worked out without adding to the length: the last 63 integers are refused like any
    # other length beyond the table, by every variant, and as the bound of the lengths the largest integer is as good as any.
    w = W.generate(W.small_config(batch=4, n_q_heads=hq, n_kv_heads=hkv, ctx=1200, n_nodes=n_nodes, paged=paged))
    ref = oracle.tree_attn(w.q, w.k_cache, w.v_cache, w.k_tree, w.v_tree, w.parent, w.ctx_len, w.scale, block_table=w.block_table)[0]
    most = 2 ** 31 - 1
    st = make_step(w)
    for bad in ([most, most - 62], [most - 63, most - 31], [-most - 1, most - 1]):
        lens = w.ctx_len.copy()
        lens[1], lens[2] = bad
        st.ctx_len.copy_(torch.from_numpy(lens))
        for bound in (1200, most):
            st.out.fill_(float("nan"))
            clv.clv_tree_attn(st.shape, st.cache, st.q, st.k_tree, st.v_tree, st.parent, st.ctx_len, bound, w.scale, st.out, st.lse,
                              st.status[0], st.workspace)
            torch.cuda.synchronize()
            assert st.status[0].cpu().tolist() == [0, clv.CLV_ERR_TREE, clv.CLV_ERR_TREE, 0]
            for b in (0, 3):
                assert_attn_close(bits(st.out)[b], ref[b], "beside lengths of %s" % bad)


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("n_nodes", [16, 50])
def test_attention_asks_ahead_by_hints_that_are_wrong(clv, oracle, n_nodes, paged):
    # Key tiles are asked for into L2 by the lengths and pages as they stand ahead of the previous kernel's end (row tiles of up to
    # 64 rows, three key tiles per block and more): lengths and pages out of range, and lengths that the commit in front changes.
    w = W.generate(W.small_config(batch=4, n_q_heads=4, n_kv_heads=4, ctx=4000, n_nodes=n_nodes, paged=paged))
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st)
    good = w.ctx_len.copy()
    alen, aidx = torch.tensor([3, 0, 2, 1], dtype=torch.int32, device="cuda"), torch.zeros(4, w.path_cap, dtype=torch.int32, device="cuda")
    aidx[:, :3] = torch.arange(3, device="cuda", dtype=torch.int32)
    before = torch.from_numpy(good - np.array([3, 0, 2, 1], np.int32)).cuda()
    moved = st.k_cache.clone(), st.v_cache.clone()
    for _ in range(3):      # the commit advances the lengths to `good` and overwrites rows that attention reads right behind it
        st.k_cache.copy_(moved[0]); st.v_cache.copy_(moved[1]); st.ctx_len.copy_(before)
        clv.clv_kv_commit(st.shape, st.cache, st.k_tree, st.v_tree, aidx, alen, st.ctx_len, st.ctx_len, st.status[2])
        st.tree_attn()
    torch.cuda.synchronize()
    assert np.array_equal(st.ctx_len.cpu().numpy(), good)
    w.k_cache[:], w.v_cache[:] = bits(st.k_cache), bits(st.v_cache)
    check_attention(oracle, w, st)
    bad = good.copy()
    bad[1], bad[2] = -5, 1 << 30
    st.ctx_len.copy_(torch.from_numpy(bad))
    flagged = [0, clv.CLV_ERR_TREE, clv.CLV_ERR_TREE, 0]
    if paged:
        table = w.block_table.copy()
        table[3, :5] = [-7, w.n_pages, 1 << 30, -1, w.n_pages + 5]
        st.block_table.copy_(torch.from_numpy(table))
        flagged[3] = clv.CLV_ERR_TREE
    st.tree_attn()
    torch.cuda.synchronize()
    assert st.status[0].cpu().tolist() == flagged


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("n_nodes", [16, 50])
def test_attention_asks_ahead_by_hints_of_other_tiles(clv, oracle, n_nodes, paged):
    # The kernel in front of attention writes the lengths, or the block table: what stands there until then is a length pages and
    # splits away (or none), pages of other sequences or none.  A commit of empty paths writes its input's lengths to another
    # array and lets the next kernel be set up meanwhile, so attention's hints are the old words.
    w = W.generate(W.small_config(batch=4, n_q_heads=4, n_kv_heads=4, ctx=4000, n_nodes=n_nodes, paged=paged))
    st = make_step(w)
    w.ctx_len[:] = [191, 1281, 4000, 2048]
    ref = oracle.tree_attn(w.q, w.k_cache, w.v_cache, w.k_tree, w.v_tree, w.parent, w.ctx_len, w.scale, block_table=w.block_table)[0]

    def writer(words, out):   # a commit that leaves `words` in `out`
        n = words.size
        src, zero = torch.from_numpy(np.ascontiguousarray(words.reshape(-1))).cuda(), torch.zeros(n, 1, dtype=torch.int32, device="cuda")
        tree, k, v = (torch.zeros(n, 1, 1, 128, dtype=torch.bfloat16, device="cuda") for _ in range(3))
        shape, status = clv.make_shape(n, 1, 1, 1, 1, 1), torch.zeros(n, dtype=torch.int32, device="cuda")
        return lambda: clv.clv_kv_commit(shape, clv.make_cache(k, v), tree, tree, zero, zero, src, out, status)

    real = {"lengths": (w.ctx_len, st.ctx_len)}
    stale = {"lengths": [[4000, 1, 0, 3841], [0, 4000, 63, 4000], [-1, 2 ** 31 - 1, 1 << 30, 65]]}
    if paged:
        real["pages"] = (w.block_table, st.block_table)
        stale["pages"] = [np.roll(w.block_table, 1, axis=0), np.full_like(w.block_table, -1), np.full_like(w.block_table, w.n_pages),
                          w.block_table[:, ::-1]]
    put = {name: writer(words.astype(np.int32), out) for name, (words, out) in real.items()}
    for last in real:
        for old in stale[last]:
            for name, (words, out) in real.items():
                out.copy_(torch.from_numpy(np.ascontiguousarray(words)))
            real[last][1].copy_(torch.from_numpy(np.ascontiguousarray(np.int32(old))))
            st.out.fill_(float("nan"))
            put[last]()
            st.tree_attn()
            torch.cuda.synchronize()
            assert st.status[0].cpu().tolist() == [0, 0, 0, 0]
            assert np.array_equal(st.ctx_len.cpu().numpy(), w.ctx_len)
            assert_attn_close(bits(st.out), ref, "%s of %s" % (last, old))


@pytest.mark.parametrize("paged", [False, True])
def test_attention_units_of_many_row_tiles(clv, oracle, paged):
    # four row tiles per (sequence, kv head) (GQA 4 x 128 nodes = 512 rows): such units are worked
    # by blocks of two row tiles; ragged contexts, one of them shorter than a key tile, key splits
    cfg = W.small_config(batch=3, n_q_heads=8, n_kv_heads=2, ctx=(50, 1300), n_nodes=128, vocab=64,
                         paged=paged, seed=W.BASE_SEED + 512)
    w = W.generate(cfg)
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st)


@pytest.mark.parametrize("batch,hq,hkv,ctx,n_nodes", [
    (5, 8, 8, (130, 700), 20),      # 40 units: the keys of a unit over 3 blocks
    (3, 8, 8, (64, 1200), 33),      # 24 units: over 5
    (11, 2, 2, (1, 900), 40),       # 22 units: over 6
    (1, 15, 15, (2050, 2050), 65),  # 15 units: over 7 or 8, an odd number of tiles
    (7, 32, 8, (60, 390), 96),      # three row tiles per unit and more units than half the machine: two per block
])
def test_attention_splits_and_row_tiles(clv, oracle, batch, hq, hkv, ctx, n_nodes):
    cfg = W.small_config(batch=batch, n_q_heads=hq, n_kv_heads=hkv, ctx=ctx, n_nodes=n_nodes, vocab=64,
                         seed=W.BASE_SEED + 31 * batch)
    w = W.generate(cfg)
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st)


@pytest.mark.parametrize("hq,hkv,n_nodes,ctx", [
    (4, 4, 32, (0, 70)),        # 32 rows, four threads per row; one or two tiles, some parts without a key
    (16, 16, 33, (190, 2100)),  # 33 rows, two threads per row
    (14, 2, 4, (100, 600)),     # 28 rows of a group of 7: rows of a copy that no node has
    (14, 2, 9, (65, 1300)),     # 63 rows
    (2, 2, 64, (4000, 9000)),   # 64 rows, the keys over all blocks of a cluster
    (1, 1, 1, (1, 40)),         # one row
])
def test_attention_rows_shared_by_threads(clv, oracle, hq, hkv, n_nodes, ctx):
    cfg = W.small_config(batch=3, n_q_heads=hq, n_kv_heads=hkv, ctx=ctx, n_nodes=n_nodes, vocab=64,
                         paged=n_nodes == 33, seed=W.BASE_SEED + 700 + n_nodes)
    w = W.generate(cfg)
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st)


@pytest.mark.parametrize("n_nodes,hq,batch", [
    (13, 8, 40),    # 13 rows, four threads per row
    (33, 8, 40),    # 33 rows, two threads per row
    (48, 16, 30),   # 96 rows, one thread per row
])
def test_attention_of_a_block_alone_rounds_once(clv, oracle, n_nodes, hq, batch):
    # More units than the machine takes at a time, so no unit's keys are shared out over blocks and
    # nothing but the output is rounded to 16 bits.  With equal scores and whole values every
    # probability and sum is exact in fp32; the quotient is within a few 2^-24, so the output is the
    # bf16 number nearest to the exact mean, except where that lies within 2^-20 of a midpoint.
    cfg = W.small_config(batch=batch, n_q_heads=hq, n_kv_heads=8, ctx=(90, 300), n_nodes=n_nodes, vocab=64,
                         seed=W.BASE_SEED + 811 + n_nodes)
    w = W.generate(cfg)
    rng = np.random.default_rng(811)
    w.q[:] = 0
    for name in ("v_cache", "v_tree"):
        v = rng.integers(1, 256, size=getattr(w, name).shape).astype(np.float32)
        setattr(w, name, W.f32_to_bf16_bits(v))
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    ref = check_attention_status(oracle, w, st)
    nearest = [W.f32_to_bf16_bits((ref * (1 + d)).astype(np.float32)) for d in (-2.0 ** -20, 2.0 ** -20)]
    got, sure = bits(st.out), nearest[0] == nearest[1]
    assert sure.mean() > 0.99
    assert np.array_equal(got[sure], nearest[0][sure])


@pytest.mark.parametrize("n_nodes", [16, 128])
def test_attention_scores_that_outgrow_the_first_tile(clv, oracle, n_nodes):
    # Keys 128 times larger from position 300 on: scores rise by far more than 2^32 between the tiles,
    # so the running reference of a row is replaced and its accumulator rescaled.  Scores reach about
    # 500, where float32 resolves 6e-5: within the tolerance of the check.
    cfg = W.small_config(batch=2, n_q_heads=8, n_kv_heads=2, ctx=(500, 1400), n_nodes=n_nodes, vocab=64,
                         seed=W.BASE_SEED + 606)
    w = W.generate(cfg)
    w.k_cache[:, 300:] = _scale_bf16_by_pow2(w.k_cache[:, 300:], 7)
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st)


def judges_of_a_tile(w, tile, slots_share_keys):
    """What the kernel's softmax judges a row's reference by at one key tile of the context, in float64: the sum of the
    first 64 keys' probabilities, and the largest of the other 64 in log2 units above the reference.  A block that is
    alone walks all tiles of its unit (with two row tiles per block), or every second one (one row tile, two slots)."""
    B, N, Hq, D = w.q.shape
    G = Hq // w.cfg.n_kv_heads
    q, k = W.bf16_bits_to_f64(w.q), W.bf16_bits_to_f64(w.k_cache[:, :(tile + 1) * 128])
    s = np.einsum("bnhd,bkhd->bnhk", q, np.repeat(k, G, axis=2), optimize=True) * (w.scale * np.log2(np.e))
    ref = None
    for t in range(tile % 2 if slots_share_keys else 0, tile + 1, 2 if slots_share_keys else 1):
        x = s[..., t * 128:(t + 1) * 128]
        if ref is None:
            ref = x.max(-1)
            continue
        with np.errstate(over="ignore"):
            total = np.exp2(x[..., :64] - ref[..., None]).sum(-1)
        above = x[..., 64:].max(-1) - ref
        if t < tile:   # nothing happens before the tile in question
            assert total.max() < 256 and above.max() < 8
    return s[..., tile * 128:], ref, total, above


@pytest.mark.parametrize("n_nodes,tile,key", [
    (64, 2, 0), (64, 2, 32), (64, 2, 63), (64, 2, 96),       # one row tile: the first slot,
    (64, 3, 31), (64, 3, 64), (64, 3, 127),                  #   the second
    (128, 3, 0), (128, 3, 63), (128, 3, 64), (128, 3, 95),   # two row tiles per block
])
def test_attention_reference_replaced_in_every_part_of_a_tile(clv, oracle, n_nodes, tile, key):
    # Blocks are alone and take two to five tiles per slot.  In one tile behind a slot's first, one key is 128 times as
    # large, so that about half of the rows' scores outgrow their reference by up to 2^700, and one judge only sees it: the
    # sum for a tile's first 64 keys, the maximum for the others.  fp32 resolves such scores within the tolerance.
    cfg = W.small_config(batch=40, n_q_heads=8, n_kv_heads=4, ctx=(520, 640), n_nodes=n_nodes, vocab=64,
                         seed=W.BASE_SEED + 640 + key)
    w = W.generate(cfg)
    at = tile * 128 + key
    w.k_cache[:, at] = _scale_bf16_by_pow2(w.k_cache[:, at], 7)
    _, _, total, above = judges_of_a_tile(w, tile, slots_share_keys=n_nodes == 64)
    by_sum, by_max = total > 256, above > 8
    assert (by_sum if key < 64 else by_max).mean() > 0.4 and not (by_max if key < 64 else by_sum).any()
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st)


@pytest.mark.parametrize("n_nodes,tile", [(64, 2), (64, 3), (128, 3)])
def test_attention_reference_replaced_for_the_sum_alone(clv, oracle, n_nodes, tile):
    # The first 64 keys of a tile are all about 2^6.5 above the rows' references: none reaches 2^8, their sum is
    # about 2^12.  Values are positive and reach 2^118, so an accumulator against the old references would overflow.
    cfg = W.small_config(batch=40, n_q_heads=8, n_kv_heads=4, ctx=(520, 640), n_nodes=n_nodes, vocab=64, seed=W.BASE_SEED + 648)
    w = W.generate(cfg)
    w.q[:] = _scale_bf16_by_pow2(w.q, -3)
    w.q[..., 0] = W.f32_to_bf16_bits(np.float32([8.0]))[0]
    w.k_cache[..., 0] = w.k_tree[..., 0] = 0
    w.k_cache[:, tile * 128:tile * 128 + 64, :, 0] = W.f32_to_bf16_bits(np.float32([7 / (8 * w.scale * np.log2(np.e))]))[0]
    rng = np.random.default_rng(648)
    for name in ("v_cache", "v_tree"):
        v = rng.uniform(1.0, 2.0, size=getattr(w, name).shape).astype(np.float32) * np.float32(2.0 ** 117)
        setattr(w, name, W.f32_to_bf16_bits(v))
    scores, ref, total, above = judges_of_a_tile(w, tile, slots_share_keys=n_nodes == 64)
    assert (scores[..., :64].max(-1) - ref).max() < 8 and above.max() < 8 and total.min() > 2.0 ** 11.9
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    want = check_attention_status(oracle, w, st)
    got = bits(st.out)
    assert np.isfinite(W.bf16_bits_to_f64(got)).all()
    _, rel = attn_errors(got, want)
    assert rel <= ATTN_MAX_REL, rel


@pytest.mark.parametrize("batch,hq,hkv,ctx,n_nodes", [
    (20, 16, 4, (40, 900), 33),    # two row tiles per block
    (20, 8, 4, (40, 900), 100),
    (44, 8, 2, (10, 700), 70),     # one
])
def test_attention_ragged_batches_in_a_small_pool(clv, oracle, batch, hq, hkv, ctx, n_nodes):
    # blocks of very unequal lengths, several to an SM
    cfg = W.small_config(batch=batch, n_q_heads=hq, n_kv_heads=hkv, ctx=ctx, n_nodes=n_nodes, vocab=64, paged=True,
                         seed=W.BASE_SEED + 660 + batch)
    w = W.generate(cfg)
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st)


@pytest.mark.parametrize("batch,hq,hkv,ctx,n_nodes", [
    (20, 8, 4, (60, 2500), 64),    # 80 units on 148 SMs: blocks are alone, partial sums stay fp32
    (20, 8, 4, (60, 2500), 100),
    (10, 16, 4, (60, 2500), 42),
    (20, 16, 4, (40, 900), 33),
    (44, 8, 2, (10, 700), 70),
])
def test_attention_of_a_paged_batch_whatever_the_pool(clv, oracle, batch, hq, hkv, ctx, n_nodes):
    # The size of a pool says nothing about a batch's lengths: it may hold other batches' pages, and sequences may
    # share theirs.  So the same bits come from a pool that just holds the batch and from one of three times the pages.
    cfg = W.small_config(batch=batch, n_q_heads=hq, n_kv_heads=hkv, ctx=ctx, n_nodes=n_nodes, vocab=64, paged=True,
                         seed=W.BASE_SEED + 680 + batch)
    w = W.generate(cfg)
    st = make_step(w)
    st.tree_attn()
    w.k_cache, w.v_cache = (np.concatenate([c, c[::-1], c]) for c in (w.k_cache, w.v_cache))
    st2 = make_step(w)
    st2.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st2)
    assert torch.equal(st.out, st2.out) and torch.equal(st.lse, st2.lse) and torch.equal(st.status[0], st2.status[0])


@pytest.mark.parametrize("batch,hq,hkv,n_nodes", [(20, 8, 4, 64), (16, 32, 8, 64), (12, 4, 4, 20), (3, 8, 2, 128)])
def test_attention_with_shared_pages_and_a_loose_bound(clv, oracle, batch, hq, hkv, n_nodes):
    # Every sequence begins with the same seven pages, and the bound is eight times the longest context, in a
    # pool of a few pages per sequence.
    cfg = W.small_config(batch=batch, n_q_heads=hq, n_kv_heads=hkv, ctx=(448, 700), n_nodes=n_nodes, vocab=64, paged=True,
                         seed=W.BASE_SEED + 690 + batch)
    w = W.generate(cfg)
    w.block_table[:, :7] = w.block_table[0, :7]
    used, w.block_table = np.unique(w.block_table, return_inverse=True)   # the pages that are left, numbered anew
    w.block_table = w.block_table.reshape(batch, -1).astype(np.int32) - (1 if used[0] < 0 else 0)
    w.k_cache, w.v_cache = (np.ascontiguousarray(c[used[used >= 0]]) for c in (w.k_cache, w.v_cache))
    for bound in (1, 8):
        st = make_step(w)
        st.max_ctx_len *= bound
        st.tree_attn()
        torch.cuda.synchronize()
        check_attention(oracle, w, st)


@pytest.mark.parametrize("batch,hq,hkv,n_nodes", [
    (2, 8, 8, 16),    # one row tile of 16 rows, of 128 (two slots share it), two row tiles per block;
    (2, 8, 2, 32),    #   keys over several blocks
    (2, 8, 2, 64),
    (40, 8, 4, 64),   # blocks alone
    (40, 4, 4, 20),
])
def test_attention_large_values_beside_rising_scores(clv, oracle, batch, hq, hkv, n_nodes):
    # Scores rise by up to about 2^40 behind the first tiles and the values reach 2^112: a probability of
    # 2^8 against the row's reference leaves room for that in an fp32 accumulator, one of 2^16 does not.
    cfg = W.small_config(batch=batch, n_q_heads=hq, n_kv_heads=hkv, ctx=(420, 900), n_nodes=n_nodes, vocab=64,
                         seed=W.BASE_SEED + 613)
    w = W.generate(cfg)
    w.k_cache[:, 300:] = _scale_bf16_by_pow2(w.k_cache[:, 300:], 3)
    for name in ("v_cache", "v_tree"):
        setattr(w, name, _scale_bf16_by_pow2(getattr(w, name), 110))
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    ref = check_attention_status(oracle, w, st)
    got = bits(st.out)
    assert np.isfinite(W.bf16_bits_to_f64(got)).all()
    _, rel = attn_errors(got, ref)
    assert rel <= ATTN_MAX_REL, rel


@pytest.mark.parametrize("batch,hq,hkv,n_nodes,ctx", [(8, 16, 16, 20, (205, 215)), (3, 32, 8, 100, (240, 430))])
def test_attention_lse_is_rounded_once(clv, oracle, batch, hq, hkv, n_nodes, ctx):
    # Relative root mean square error of the log-sum-exp.  One rounding to fp32 has at most 2^-24 / sqrt(3) =
    # 3.4e-8 (results just above a power of two); the fp32 sum of some 220 exponentials of 2^-22
    # each, with either sign, adds about 2e-8: together below 4.3e-8.  (Two roundings: 4.8e-8 to 5.4e-8.)
    cfg = W.small_config(batch=batch, n_q_heads=hq, n_kv_heads=hkv, ctx=ctx, n_nodes=n_nodes, vocab=64,
                         seed=W.BASE_SEED + 619)
    w = W.generate(cfg)
    st = make_step(w)
    st.tree_attn()
    torch.cuda.synchronize()
    lse = oracle.tree_attn(w.q, w.k_cache, w.v_cache, w.k_tree, w.v_tree, w.parent, w.ctx_len, w.scale)[2]
    err = st.lse.cpu().numpy().astype(np.float64) / lse - 1
    assert np.sqrt((err ** 2).mean()) <= 4.3e-8


@pytest.mark.parametrize("n_nodes", [24, 128])   # one row tile per block / two row tiles per block
def test_attention_wait_that_runs_out_is_reported_and_leaves_the_library_usable(clv, oracle, n_nodes):
    # Every on-chip wait of the attention kernel is bounded.  With the bound cut to a few dozen SM
    # cycles the ordinary wait for the first tile (a load from device memory takes far longer)
    # runs out: the blocks must leave in order - copies and tensor-core work in flight waited for,
    # tensor memory released - the call itself succeeds, and status[] says CLV_ERR_TIMEOUT.
    # Nothing faults; the next call, on the same workspace, is an ordinary one.
    cfg = W.small_config(batch=2, n_q_heads=8, n_kv_heads=2, ctx=(300, 700), n_nodes=n_nodes, vocab=64,
                         seed=W.BASE_SEED + 404)
    w = W.generate(cfg)
    st = make_step(w)
    try:
        clv.clv_test_set_wait_limit(32)
        st.tree_attn()
        torch.cuda.synchronize()
    finally:
        clv.clv_test_set_wait_limit(0)
    assert st.status[0].cpu().tolist() == [clv.CLV_ERR_TIMEOUT] * 2
    st.status.zero_()
    st.tree_attn()
    torch.cuda.synchronize()
    check_attention(oracle, w, st)


@pytest.mark.parametrize("batch,hq,hkv,n_nodes", [
    (3, 8, 8, 16),    # clusters: four threads per row, two, one, two row tiles
    (3, 4, 4, 60),
    (3, 8, 2, 32),
    (2, 16, 2, 128),
    (40, 8, 4, 13),   # blocks alone
    (40, 8, 2, 32),
])
def test_attention_waits_that_run_out_anywhere_are_reported(clv, oracle, batch, hq, hkv, n_nodes):
    # Bounds from below the first wait to above the last one: whichever wait runs out (for a tile, for the last
    # product, for another block's rows), a sequence whose status is CLV_OK has the right rows.
    cfg = W.small_config(batch=batch, n_q_heads=hq, n_kv_heads=hkv, ctx=(300, 2300), n_nodes=n_nodes, vocab=64,
                         seed=W.BASE_SEED + 405)
    w = W.generate(cfg)
    st = make_step(w)
    ref = oracle.tree_attn(w.q, w.k_cache, w.v_cache, w.k_tree, w.v_tree, w.parent, w.ctx_len, w.scale)[0]
    seen = set()
    for limit in [32, 200, 400, 600, 800, 1000, 1300, 1600, 2000, 2500, 3000, 4000, 6000, 9000, 20000, 100000, 0]:
        st.out.fill_(float("nan"))
        st.status.fill_(-7)
        try:
            clv.clv_test_set_wait_limit(limit)
            st.tree_attn()
            torch.cuda.synchronize()
        finally:
            clv.clv_test_set_wait_limit(0)
        status = st.status[0].cpu().numpy()
        seen.add((limit, bool(status.any())))
        assert set(status.tolist()) <= {clv.CLV_OK, clv.CLV_ERR_TIMEOUT}, limit
        done = status == clv.CLV_OK
        if done.any():
            assert_attn_close(bits(st.out)[done], ref[done], limit)
    assert (32, True) in seen and (0, False) in seen


def test_attention_waits_that_run_out_in_a_sequence_of_more_blocks_than_run_at_once(clv, oracle):
    # 149 heads in clusters of two: 298 blocks of one sequence, 148 of them at a time, so that blocks whose waits run out
    # late are gone before the last are counted.  Their failures must reach the status all the same, and promptly.
    w = W.generate(W.small_config(batch=1, n_q_heads=149, n_kv_heads=149, ctx=6000, n_nodes=16, vocab=64, seed=W.BASE_SEED + 406))
    st = make_step(w)
    rows = np.array([[0, i, h] for h in range(149) for i in (0, 15)], np.int64)
    ref = oracle.tree_attn(w.q, w.k_cache, w.v_cache, w.k_tree, w.v_tree, w.parent, w.ctx_len, w.scale, rows=rows)[0]
    for limit in [32, 400, 800, 1300, 2000, 3000, 4000, 5000, 6000, 9000, 20000, 100000, 0]:
        for _ in range(3):
            st.out.fill_(float("nan"))
            st.status.fill_(-7)
            try:
                clv.clv_test_set_wait_limit(limit)
                st.tree_attn()
                torch.cuda.synchronize()
            finally:
                clv.clv_test_set_wait_limit(0)
            status = int(st.status[0, 0])
            assert status in (clv.CLV_OK, clv.CLV_ERR_TIMEOUT) and (limit or status == clv.CLV_OK)
            if status == clv.CLV_OK:
                assert not torch.isnan(st.out).any()
                assert_attn_close(bits(st.out)[rows[:, 0], rows[:, 1], rows[:, 2]], ref, limit)


# ------------------------------------------------------------------ argmax
@pytest.mark.parametrize("vocab,ld_pad", [(1, 0), (7, 0), (8, 8), (2047, 0), (2049, 16),
                                          (32000, 0), (50257, 8), (128256, 0)])
def test_argmax_sizes(clv, oracle, vocab, ld_pad):
    rows_b, rows_n = 2, 5
    ld = (vocab + 7) // 8 * 8 + ld_pad
    rng = np.random.default_rng(vocab)
    winner = rng.integers(0, vocab, size=rows_b * rows_n)
    lg = W.make_logits(rows_b * rows_n, vocab, ld, winner, 0.5, seed=vocab + 1)
    lg[:, vocab:] = 0x7F00                  # huge values in the padding must be ignored
    shape = clv.make_shape(rows_b, rows_n, 1, 1, vocab, 1)
    ws = clv.new_workspace(shape, None, 0)
    d = torch.from_numpy(lg.view(np.int16)).cuda()
    ids = torch.empty(rows_b, rows_n, dtype=torch.int32, device="cuda")
    clv.clv_accept_argmax(shape, d, ld, ids, ws)
    clv.clv_accept_argmax(shape, d, ld, ids, ws)     # the workspace is reusable as is
    torch.cuda.synchronize()
    ref = oracle.argmax(lg, vocab)
    assert np.array_equal(ids.cpu().numpy().reshape(-1), ref)
    if vocab > 1:
        assert np.array_equal(ref, winner)


def test_argmax_ties_zeros_and_infinities(clv, oracle):
    vocab = 40000                            # several chunks per row
    cfg = W.small_config(batch=1, n_nodes=8, vocab=vocab)
    w = W.generate(cfg)
    lg = w.logits[0]
    lg[:] = W.f32_to_bf16_bits(np.full(lg.shape, -1.0, np.float32))
    one = 0x3F80
    lg[0, [39999, 17, 20000]] = one          # equal maxima in different chunks: lowest index
    lg[1, vocab - 1] = one                   # maximum in the very last column
    lg[2, 0] = one
    lg[3, :] = 0x8000                        # all -0.0 with a +0.0 later: index 0
    lg[3, 30000] = 0x0000
    lg[4, :] = 0xFF80                        # all -inf
    lg[5, 25000] = 0x0000                    # +0.0 after -0.0, both above the -1 background
    lg[5, 123] = 0x8000
    lg[6, [5, 6, 7, 4]] = one                # ties inside one 16-byte vector
    lg[7, :] = 0xFF80
    lg[7, 33333] = 0xC2C8                    # -100 among -inf
    st = make_step(w)
    st.accept_argmax()
    torch.cuda.synchronize()
    ref = oracle.argmax(w.logits, vocab)
    assert ref[0].tolist() == [17, vocab - 1, 0, 0, 0, 123, 4, 33333]
    assert np.array_equal(st.ids.cpu().numpy(), ref)


@pytest.mark.parametrize("rows_b,rows_n,vocab", [(3, 7, 40008), (1, 1, 8), (2, 64, 9000), (5, 3, 2051), (1, 128, 33)])
def test_argmax_cuts_ties_and_ragged_rows(clv, oracle, rows_b, rows_n, vocab):
    # A row is scanned in pieces by several blocks, wherever the cuts fall: equal maxima planted far
    # apart (first index wins), maxima in the ragged last elements of a row (vocab not a multiple
    # of 8), and a second call on the same workspace.
    ld = (vocab + 7) // 8 * 8 + 8
    rng = np.random.default_rng(vocab * 31 + rows_n)
    rows = rows_b * rows_n
    lg = np.empty((rows, ld), np.uint16)
    lg[:] = W.f32_to_bf16_bits(rng.standard_normal((rows, ld)).astype(np.float32))
    big = int(W.f32_to_bf16_bits(np.array([9.0], np.float32))[0])
    for r in range(rows):
        k = r % 4
        if k == 0:
            pos = sorted(set(int(x) for x in rng.integers(0, vocab, size=5)))
            lg[r, pos] = big                      # ties far apart
        elif k == 1:
            lg[r, vocab - 1] = big                # the very last (possibly ragged) element
        elif k == 2:
            lg[r, max(0, vocab - 3)] = big
            lg[r, vocab // 2] = big               # tie between the middle and the ragged end
        # k == 3: plain random row
    lg[:, vocab:] = 0x7F00                        # huge values in the padding must be ignored
    shape = clv.make_shape(rows_b, rows_n, 1, 1, vocab, 1)
    ws = clv.new_workspace(shape, None, 0)
    d = torch.from_numpy(lg.view(np.int16)).cuda()
    ids = torch.full((rows_b, rows_n), -5, dtype=torch.int32, device="cuda")
    ref = oracle.argmax(lg, vocab)
    for _ in range(2):
        clv.clv_accept_argmax(shape, d, ld, ids, ws)
        torch.cuda.synchronize()
        assert np.array_equal(ids.cpu().numpy().reshape(-1), ref)
        ids.fill_(-5)


@pytest.mark.parametrize("rows,vocab", [(1, 262144), (1, 262153), (74, 153600), (74, 153601), (75, 196608), (110, 196615), (111, 196609), (3, 100003), (74, 2051), (75, 2051), (148, 4100), (149, 32768), (149, 32776), (149, 57344), (296, 57345),
                                        (296, 32769), (297, 8195), (592, 6147), (593, 6147), (600, 8193)])
def test_argmax_at_the_edges_of_its_blocks(clv, oracle, rows, vocab):
    # How a row is shared depends on rows and vocabulary (148 SMs): both sides of every line, with remainders of the
    # batches of loads.  Ties: a maximum in the last element and one anywhere before it.
    ld = (vocab + 7) // 8 * 8 + 8
    rng = np.random.default_rng(vocab + rows)
    lg = np.empty((rows, ld), np.uint16)
    lg[:, :vocab] = W.f32_to_bf16_bits(rng.standard_normal(vocab + 131).astype(np.float32))[np.arange(vocab) + np.arange(rows)[:, None] % 131]
    lg[:, vocab:] = 0x7F00                        # huge values in the padding must be ignored
    big = int(W.f32_to_bf16_bits(np.array([9.0], np.float32))[0])
    lg[:, vocab - 1] = big
    at = rng.integers(0, vocab, size=rows)
    lg[np.arange(rows)[::2], at[::2]] = big
    shape = clv.make_shape(rows, 1, 1, 1, vocab, 1)
    ids = torch.full((rows, 1), -5, dtype=torch.int32, device="cuda")
    clv.clv_accept_argmax(shape, torch.from_numpy(lg.view(np.int16)).cuda(), ld, ids, clv.new_workspace(shape, None, 0))
    torch.cuda.synchronize()
    ref = oracle.argmax(lg, vocab)
    assert np.array_equal(ref[::2], at[::2]) and (ref[1::2] == vocab - 1).all()
    assert np.array_equal(ids.cpu().numpy().reshape(-1), ref)


def argmax_time(clv, rows, vocab):
    """Shortest time of a call among others, in ms, over logits that change from call to call."""
    ld, calls = (vocab + 7) // 8 * 8, 24
    sets = max(2, min(calls, (1 << 28) // (2 * rows * ld)))
    lg = torch.randn(sets, rows, ld, dtype=torch.bfloat16, device="cuda")
    shape = clv.make_shape(rows, 1, 1, 1, vocab, 1)
    ids, ws = torch.zeros(rows, 1, dtype=torch.int32, device="cuda"), clv.new_workspace(shape, None, 0)
    clv.clv_accept_argmax(shape, lg[0], ld, ids, ws)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for k in range(calls):
            clv.clv_accept_argmax(shape, lg[k % sets], ld, ids, ws)
    best = 1e9
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        g.replay()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / calls)
    return best


@pytest.mark.parametrize("rows,others", [(22, 25), (23, 25), (24, 25), (47, 50), (48, 50), (49, 50), (72, 66), (74, 66)])
def test_argmax_has_no_last_cluster_that_waits_for_a_wave(clv, rows, others):
    # Clusters of six fill a GPU's parts only so far: a grid whose blocks were shared out evenly over all SMs took up to 1.7 times
    # what a few rows more or less took.  The bound is what the rows' number explains and a quarter.
    assert argmax_time(clv, rows, 128256) <= 1.25 * max(1.0, rows / others) * argmax_time(clv, others, 128256)


@pytest.mark.parametrize("rows,vocab,other_rows,other_vocab", [(4, 200000, 4, 262152), (25, 262144, 25, 262152), (75, 1 << 20, 74, 1 << 20)])
def test_argmax_takes_no_longer_for_fewer_logits(clv, rows, vocab, other_rows, other_vocab):
    # a few long rows are cut finely enough to fill the GPU: whole rows and clusters of six left half of it idle (1.2 to 1.4 times)
    assert argmax_time(clv, rows, vocab) <= 1.1 * argmax_time(clv, other_rows, other_vocab)


# ------------------------------------------------------------------ walk and commit
def test_walk_random_trees_and_errors(clv, oracle):
    rng = np.random.default_rng(5)
    B, N = 64, 48
    cfg = W.small_config(batch=B, n_nodes=N, vocab=16, n_q_heads=1, n_kv_heads=1, ctx=1)
    w = W.generate(cfg)
    tokens = np.stack([W._draw_tokens(w.parent[b], 64, rng) for b in range(B)])
    ids = np.stack([W._plant_winners(w.parent[b], tokens[b], 64, 0.7, rng) for b in range(B)])
    w.parent[3, 0] = 0                        # root is not a root
    w.parent[4, 9] = -1                       # second root
    w.parent[5, 7] = 7                        # self parent
    w.parent[6] = W.tree_chain(N)             # deep chain, every edge agreeing: overflows path_cap
    tokens[6] = np.arange(N)
    ids[6, :-1] = tokens[6, 1:]
    from paper_2408_00264_b200 import binding as b
    dev = "cuda"
    shape = b.make_shape(B, N, 1, 1, 16, 9)
    t = lambda a: torch.from_numpy(a).to(dev)
    alen = torch.empty(B, dtype=torch.int32, device=dev)
    aidx = torch.empty(B, 9, dtype=torch.int32, device=dev)
    nxt = torch.empty(B, dtype=torch.int32, device=dev)
    stt = torch.empty(B, dtype=torch.int32, device=dev)
    b.clv_accept_walk(shape, t(w.parent), t(tokens), t(ids), alen, aidx, nxt, stt)
    torch.cuda.synchronize()
    r_len, r_idx, r_nxt, r_st = oracle.accept_walk(w.parent, tokens, ids, 9)
    assert np.array_equal(alen.cpu().numpy(), r_len) and np.array_equal(aidx.cpu().numpy(), r_idx)
    assert np.array_equal(nxt.cpu().numpy(), r_nxt) and np.array_equal(stt.cpu().numpy(), r_st)
    assert r_st[[3, 4, 5, 6]].tolist() == [7, 7, 7, 7] and r_len.max() >= 2


@pytest.mark.parametrize("paged", [False, True])
def test_commit_edges_alias_and_capacity(clv, oracle, paged):
    cfg = W.small_config(batch=4, n_q_heads=8, n_kv_heads=2, ctx=(50, 140), n_nodes=12, vocab=64,
                         paged=paged, p_accept=0.9)
    w = W.generate(cfg)
    ids = oracle.argmax(w.logits, 64)
    alen, aidx, _, _ = oracle.accept_walk(w.parent, w.tokens, ids, w.path_cap)
    alen = alen.copy()
    aidx = aidx.copy()
    ctx = w.ctx_len.copy()
    alen[1] = 0                                # nothing to commit
    if paged:
        ctx[2] = w.block_table.shape[1] * 64 - 1   # second accepted row has no page
    else:
        ctx[2] = w.cap_tokens - 1                  # second accepted row has no slot
    alen[2] = max(2, alen[2]); aidx[2, :2] = [0, 1]
    aidx[3, 0] = 12                            # node index outside the tree
    st = make_step(w)
    st.ctx_len.copy_(torch.from_numpy(ctx))
    st.accept_len.copy_(torch.from_numpy(alen))
    st.accept_idx.copy_(torch.from_numpy(aidx))
    st.kv_commit(ctx_len_out=st.ctx_len)       # in place: ctx_len_out aliases ctx_len
    torch.cuda.synchronize()
    kc, vc, new_len, s2 = oracle.kv_commit(w.k_cache, w.v_cache, w.k_tree, w.v_tree, aidx, alen,
                                           ctx, block_table=w.block_table)
    assert s2.tolist() == [0, 0, 7, 7]
    assert np.array_equal(st.ctx_len.cpu().numpy(), new_len)
    assert np.array_equal(st.status[2].cpu().numpy(), s2)
    assert np.array_equal(bits(st.k_cache), kc) and np.array_equal(bits(st.v_cache), vc)


@pytest.mark.parametrize("paged", [False, True])
def test_walk_commit_in_one_launch_with_errors(clv, oracle, paged):
    # malformed trees, a path longer than path_cap and a cache without room: the fused call gives
    # what the two calls give, sequence by sequence, and what the checker gives
    cfg = W.small_config(batch=6, n_q_heads=4, n_kv_heads=2, ctx=(10, 200), n_nodes=20, vocab=64,
                         paged=paged, seed=W.BASE_SEED + 31)
    w = W.generate(cfg)
    w.parent[1, 5] = 7            # parent after child
    w.parent[2, 0] = 0            # root is not a root
    w.parent[3, 4] = -1           # a second root: the walk refuses, attention would not
    if paged:
        w.block_table[4, :] = -1                 # sequence 4 has no page for its accepted rows
    else:
        w.ctx_len[4] = w.cap_tokens              # ... or no room left in its cache rows
    results = []
    for fused in (True, False):
        st = make_step(w)
        st.accept_argmax()
        if fused:
            st.accept_walk_commit()
        else:
            st.accept_walk()
            st.kv_commit()
        torch.cuda.synchronize()
        results.append(st)
    a, b = results
    for name in ("accept_len", "accept_idx", "next_token", "ctx_len_out", "k_cache", "v_cache"):
        assert torch.equal(getattr(a, name), getattr(b, name)), name
    assert torch.equal(a.status[1:], b.status[1:])
    ids = oracle.argmax(w.logits, w.cfg.vocab)
    alen, aidx, nxt, s1 = oracle.accept_walk(w.parent, w.tokens, ids, w.path_cap)
    kc, vc, new_len, s2 = oracle.kv_commit(w.k_cache, w.v_cache, w.k_tree, w.v_tree, aidx, alen, w.ctx_len,
                                           block_table=w.block_table)
    assert np.array_equal(a.accept_len.cpu().numpy(), alen) and np.array_equal(a.accept_idx.cpu().numpy(), aidx)
    assert np.array_equal(a.status[1].cpu().numpy(), s1) and np.array_equal(a.status[2].cpu().numpy(), s2)
    assert np.array_equal(a.ctx_len_out.cpu().numpy(), new_len)
    assert np.array_equal(bits(a.k_cache), kc) and np.array_equal(bits(a.v_cache), vc)
    assert s1.tolist()[1:4] == [7, 7, 7] and s2.tolist()[4] == 7 and s2.tolist()[0] == 0


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("n_nodes", [1, 31, 32, 33, 64, 65, 97, 128])
def test_walk_commit_at_the_edges_of_a_lane_s_nodes(clv, oracle, n_nodes, paged):
    # Sizes around the nodes that a lane holds.  Sequence 0: a chain of which every edge agrees (128 nodes from
    # position 40 on lie in three pages); 1: three tokens only, so siblings carry equal ones and the lowest
    # matching child is taken; 2: nothing agrees.
    cfg = W.small_config(batch=3, n_q_heads=4, n_kv_heads=2, ctx=40, n_nodes=n_nodes, max_depth=max(1, n_nodes - 1),
                         vocab=64, paged=paged, seed=W.BASE_SEED + 90 + n_nodes)
    w = W.generate(cfg)
    w.path_cap = n_nodes
    rng = np.random.default_rng(n_nodes)
    ids = rng.integers(0, 3, size=(3, n_nodes)).astype(np.int32)
    w.parent[0] = np.arange(n_nodes) - 1
    w.tokens[0] = np.arange(n_nodes)
    ids[0, :-1] = w.tokens[0, 1:]
    w.tokens[1] = rng.integers(0, 3, size=n_nodes)
    ids[2] = 63
    w.tokens[2] = np.minimum(w.tokens[2], 62)
    st = make_step(w)
    st.ids.copy_(torch.from_numpy(ids))
    st.accept_walk_commit()
    torch.cuda.synchronize()
    alen, aidx, nxt, s1 = oracle.accept_walk(w.parent, w.tokens, ids, w.path_cap)
    kc, vc, new_len, s2 = oracle.kv_commit(w.k_cache, w.v_cache, w.k_tree, w.v_tree, aidx, alen, w.ctx_len,
                                           block_table=w.block_table)
    assert np.array_equal(st.accept_len.cpu().numpy(), alen) and np.array_equal(st.accept_idx.cpu().numpy(), aidx)
    assert np.array_equal(st.next_token.cpu().numpy(), nxt) and np.array_equal(st.ctx_len_out.cpu().numpy(), new_len)
    assert np.array_equal(st.status[1].cpu().numpy(), s1) and np.array_equal(st.status[2].cpu().numpy(), s2)
    assert np.array_equal(bits(st.k_cache), kc) and np.array_equal(bits(st.v_cache), vc)
    assert alen[0] == n_nodes and s2.tolist() == [0, 0, 0]


def test_guard_bands_untouched(clv, oracle):
    # outputs live inside larger sentinel-filled buffers; nothing outside them may change
    cfg = W.small_config(batch=2, n_q_heads=8, n_kv_heads=2, ctx=(10, 333), n_nodes=19, vocab=4099)
    w = W.generate(cfg)
    st = make_step(w)
    pad = 4096

    def guarded(t):
        flat = torch.full((t.numel() + 2 * pad,), 0x5A5A if t.element_size() == 2 else 0x5A5A5A5A,
                          dtype=torch.int16 if t.element_size() == 2 else torch.int32,
                          device=t.device)
        inner = flat[pad: pad + t.numel()].view(t.dtype).view(t.shape)
        return flat, inner
    guards = {}
    for name in ["out", "lse", "ids", "accept_len", "accept_idx", "next_token", "ctx_len_out"]:
        g, inner = guarded(getattr(st, name))
        guards[name] = g
        setattr(st, name, inner)
    st.run()
    torch.cuda.synchronize()
    for name, g in guards.items():
        s = 0x5A5A if g.dtype == torch.int16 else 0x5A5A5A5A
        assert bool((g[:pad] == s).all()) and bool((g[-pad:] == s).all()), name
    check_attention(oracle, w, st)
    check_accept_and_commit(oracle, w, st)


def test_verify_step_from_host_buffers(clv, oracle):
    cfg = W.small_config(batch=3, n_q_heads=8, n_kv_heads=2, ctx=(20, 400), n_nodes=30, vocab=5000,
                         p_accept=0.8)
    w = W.generate(cfg)
    st = make_step(w, logits=False)
    c = w.cfg
    pin = lambda a: torch.from_numpy(a.view(np.int16) if a.dtype == np.uint16 else a).pin_memory()
    hq, hk, hv = pin(w.q), pin(w.k_tree), pin(w.v_tree)
    hp, ht, hl = pin(w.parent), pin(w.tokens), pin(w.logits)
    B, N = c.batch, c.n_nodes
    o_out = torch.empty(B, N, c.n_q_heads, 128, dtype=torch.int16).pin_memory()
    o_ids = torch.empty(B, N, dtype=torch.int32).pin_memory()
    o_len = torch.empty(B, dtype=torch.int32).pin_memory()
    o_idx = torch.empty(B, w.path_cap, dtype=torch.int32).pin_memory()
    o_nxt = torch.empty(B, dtype=torch.int32).pin_memory()
    o_st = torch.empty(3, B, dtype=torch.int32).pin_memory()
    hin = clv.ClvHostInputs(hq.data_ptr(), hk.data_ptr(), hv.data_ptr(), hp.data_ptr(),
                            ht.data_ptr(), hl.data_ptr(), w.logits.shape[-1])
    hout = clv.ClvHostOutputs(o_out.data_ptr(), o_ids.data_ptr(), o_len.data_ptr(),
                              o_idx.data_ptr(), o_nxt.data_ptr(), o_st.data_ptr())
    staging = torch.empty(clv.clv_staging_bytes(st.shape, w.logits.shape[-1]), dtype=torch.uint8,
                          device="cuda")
    clv.clv_verify_step_host(st.shape, st.cache, hin, hout, st.ctx_len, st.max_ctx_len, st.scale,
                             staging, st.workspace)
    torch.cuda.synchronize()
    ref = oracle.tree_attn(w.q, w.k_cache, w.v_cache, w.k_tree, w.v_tree, w.parent, w.ctx_len,
                           w.scale)[0]
    assert_attn_close(o_out.numpy().view(np.uint16), ref, "host step")
    ids = oracle.argmax(w.logits, c.vocab)
    alen, aidx, nxt, _ = oracle.accept_walk(w.parent, w.tokens, ids, w.path_cap)
    assert np.array_equal(o_ids.numpy(), ids) and np.array_equal(o_len.numpy(), alen)
    assert np.array_equal(o_idx.numpy(), aidx) and np.array_equal(o_nxt.numpy(), nxt)
    assert (o_st.numpy() == 0).all()
    kc, vc, new_len, _ = oracle.kv_commit(w.k_cache, w.v_cache, w.k_tree, w.v_tree, aidx, alen,
                                          w.ctx_len)
    assert np.array_equal(st.ctx_len.cpu().numpy(), new_len)
    assert np.array_equal(bits(st.k_cache), kc) and np.array_equal(bits(st.v_cache), vc)


_FIRST_CALLS = """
import sys, threading
import torch
from paper_2408_00264_b200 import binding as clv, workloads as W
from paper_2408_00264_b200.step import VerifyStep
torch.cuda.init()
steps = [VerifyStep(W.generate(W.small_config(seed=W.BASE_SEED + i))) for i in range(8)]
clv._load_calls()
torch.cuda.synchronize()
gate, failures = threading.Barrier(len(steps)), []
def first(st):
    try:
        gate.wait(60)
        st.tree_attn(torch.cuda.current_stream())
    except Exception as e:
        failures.append(repr(e))
threads = [threading.Thread(target=first, args=(st,)) for st in steps]
[t.start() for t in threads]
[t.join() for t in threads]
torch.cuda.synchronize()
assert not failures, failures
assert all(int(st.status[0].abs().sum()) == 0 for st in steps)
"""


def test_first_calls_of_a_process_from_several_threads(clv):
    # What a process sets up once (the driver's tensor-map encoder, the kernels' attributes) is set up by
    # whichever thread comes first, and the others wait for it; and a thread that has made no call of the
    # runtime before has no current context: none is refused.
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    for _ in range(3):
        subprocess.run([sys.executable, "-c", _FIRST_CALLS], check=True, cwd=root, timeout=120)


class HostCaller:
    """A small step from host buffers with its expected results; `clear` marks every result."""

    def __init__(self, clv, oracle, seed, pinned=True, shift=0):
        cfg = W.small_config(batch=2, n_q_heads=4, n_kv_heads=2, ctx=(20, 300), n_nodes=20, vocab=3000,
                             p_accept=0.8, seed=W.BASE_SEED + seed)
        w = W.generate(cfg)
        self.clv, self.st = clv, make_step(w, logits=False)
        place = (lambda t: t.pin_memory()) if pinned else (lambda t: t)
        self.host = [place(torch.from_numpy(a.view(np.int16) if a.dtype == np.uint16 else a))
                     for a in (w.q, w.k_tree, w.v_tree, w.parent, w.tokens, w.logits)]
        n = (2, 20)
        self.dst = [(place(torch.zeros(np.prod(shape) * dtype.itemsize + shift, dtype=torch.uint8)), shape, dtype)
                    for shape, dtype in (((*n, 4, 128), torch.int16), (n, torch.int32), ((2,), torch.int32),
                                         ((2, w.path_cap), torch.int32), ((2,), torch.int32), ((3, 2), torch.int32))]
        self.shift = shift   # bytes from the buffers' starts to the results
        self.hin = clv.ClvHostInputs(*[t.data_ptr() for t in self.host], w.logits.shape[-1])
        self.hout = clv.ClvHostOutputs(*[d.data_ptr() + shift for d, _, _ in self.dst])
        self.staging = torch.empty(clv.clv_staging_bytes(self.st.shape, w.logits.shape[-1]), dtype=torch.uint8, device="cuda")
        self.start = self.st.ctx_len.clone()
        ids = oracle.argmax(w.logits, w.cfg.vocab)
        self.expected = (ids, *oracle.accept_walk(w.parent, w.tokens, ids, w.path_cap)[:3])
        self.out = oracle.tree_attn(w.q, w.k_cache, w.v_cache, w.k_tree, w.v_tree, w.parent, w.ctx_len, w.scale)[0]

    def clear(self):
        for d, _, _ in self.dst:
            d.fill_(0xF9)
        self.staging.fill_(0x55)

    def step(self):
        st = self.st
        st.ctx_len.copy_(self.start)
        self.clv.clv_verify_step_host(st.shape, st.cache, self.hin, self.hout, st.ctx_len, st.max_ctx_len, st.scale,
                                      self.staging, st.workspace)

    def check(self):
        res = [d[self.shift:].clone().view(dtype).view(shape).numpy() for d, shape, dtype in self.dst]
        assert_attn_close(res[0].view(np.uint16), self.out)
        for got, ref in zip(res[1:5], self.expected):
            assert np.array_equal(got.reshape(-1), np.asarray(ref).reshape(-1))
        assert (res[5] == 0).all()


@pytest.mark.parametrize("mode", ["pageable", "unaligned", "captured", "threads"])
def test_host_step_ways_to_copy(clv, oracle, mode):
    # Pageable results and pinned ones at odd multiples of two bytes (a copy per array), a capture (no second
    # stream), a dozen threads that step at the same time; the results of every step are marked before it.
    callers = [HostCaller(clv, oracle, 900 + i, pinned=mode != "pageable", shift=2 * (mode == "unaligned"))
               for i in range(12 if mode == "threads" else 1)]
    if mode == "captured":
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            callers[0].step()
            side.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=side):
                callers[0].step()
        for _ in range(2):
            callers[0].clear()
            g.replay()
            torch.cuda.synchronize()
            callers[0].check()
        return
    torch.cuda.synchronize()
    gate, failures = threading.Barrier(len(callers)), []

    def work(c):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(12):
                    c.clear()
                    gate.wait(60)
                    c.step()
                    s.synchronize()
                    c.check()
        except BaseException as e:  # noqa: B036
            failures.append(e)
            gate.abort()
    threads = [threading.Thread(target=work, args=(c,)) for c in callers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures


@pytest.mark.parametrize("held", [1, 11])   # 11: more than the library has second streams
def test_host_steps_of_different_streams_do_not_wait_for_each_other(clv, oracle, held):
    # Steps on streams that are busy with something else for a while, then one on a free stream: that one is
    # done first.  Two steps per held stream: the second follows the first wherever its copies travel.
    # The device has eight queues for all streams, and a stream that shares one with a held stream waits
    # whatever the library does, so a few are tried (with 11 held ones only the results count).
    callers = [HostCaller(clv, oracle, 930 + i) for i in range(held + 1)]
    overtook = 0
    for attempt in range(9 if held == 1 else 2):   # the first time everything is made and loaded
        done = [torch.cuda.Event() for _ in callers]
        free, *streams = [torch.cuda.Stream() for _ in callers]
        for c in callers:
            c.clear()
        torch.cuda.synchronize()
        for c, s, e in zip(callers[:held], streams, done):
            with torch.cuda.stream(s):
                torch.cuda._sleep(300_000_000)   # about 0.15 s
                c.step()
                c.step()
                e.record()
        with torch.cuda.stream(free):
            callers[held].step()
            done[held].record()
        done[held].synchronize()
        overtook += not any(e.query() for e in done[:held])
        callers[held].check()
        torch.cuda.synchronize()
        for c in callers:
            c.check()
    assert overtook or held > 1


def test_host_step_with_a_bad_argument_leaves_the_stream_empty(clv, oracle):
    # a stride the argmax refuses: the call must fail before its first copy, so neither the
    # staging area nor the device-side context lengths change
    cfg = W.small_config(batch=2, n_q_heads=4, n_kv_heads=2, ctx=(20, 100), n_nodes=10, vocab=1000)
    w = W.generate(cfg, ld_pad=4)                       # ld = 1004, not a multiple of 8
    st = make_step(w, logits=False)
    pin = lambda a: torch.from_numpy(a.view(np.int16) if a.dtype == np.uint16 else a).pin_memory()
    host = [pin(x) for x in (w.q, w.k_tree, w.v_tree, w.parent, w.tokens, w.logits)]
    hin = clv.ClvHostInputs(*[t.data_ptr() for t in host], w.logits.shape[-1])
    outs = [torch.zeros(4096, dtype=torch.int32).pin_memory() for _ in range(6)]
    hout = clv.ClvHostOutputs(*[t.data_ptr() for t in outs])
    staging = torch.full((clv.clv_staging_bytes(st.shape, w.logits.shape[-1]),), 0x5A, dtype=torch.uint8,
                         device="cuda")
    ctx_before = st.ctx_len.clone()
    code = clv.clv_verify_step_host(st.shape, st.cache, hin, hout, st.ctx_len, st.max_ctx_len, st.scale,
                                    staging, st.workspace, check=False)
    torch.cuda.synchronize()
    assert code == clv.CLV_ERR_ALIGN
    assert bool((staging == 0x5A).all()) and torch.equal(st.ctx_len, ctx_before)
    assert all(int(t.abs().sum()) == 0 for t in outs)

"""The tiled form of chunked-prefill attention where its work split changes, against the CPU oracle: several segments of rows,
several groups of query blocks, an odd number of KV heads, repeated positions, a block of one tile beside a block of two; values of
any size, output types, score scales; and the calls that run as decode passes instead.
Bars as for every attention test (max-abs 2e-3, relative L2 1e-3) where no other is stated."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_04411_b200 import workloads
from tests.helpers import GpuCache, attn_errors, bits16
from tests.test_gpu_prefill import MAX_ABS, REL_L2, B, _case, _oracle_prefill

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hkv,rep,dtype,n_seq,ctx,n_q,repeat", [
    (1, 8, torch.float16, 1, 9000, 33, 1),       # more rows than one segment holds, a lone query in the second block
    (1, 8, torch.float16, 1, 200, 1100, 1),      # more blocks of queries than the partial results have room for
    (3, 1, torch.bfloat16, 2, 300, 150, 1),      # 384 channels: one head per reconstruction slab, six classes
    (2, 2, torch.float16, 3, 260, 65, 2),        # every position held by two tokens
    (8, 4, torch.float16, 2, 129, 4, 1),         # few queries: several splits
    (2, 4, torch.bfloat16, 1, 100, 50, 1),       # one split of one segment is the whole result
])
def test_tiled_prefill_where_the_work_split_changes(B, hkv, rep, dtype, n_seq, ctx, n_q, repeat):
    d = hkv * 128
    li = workloads.build_layer(840 + ctx, n_seq=n_seq, ctx=ctx, n_q_heads=hkv * rep, n_kv_heads=hkv, dtype=dtype, n_calib=2 * d, outlier="pct:1",
                               mode="forced", rank_recipe="any", shuffle_positions=True)
    li.positions = li.positions // repeat
    ranks = li.ranks.numpy().astype(np.int64)
    rng = np.random.default_rng(ctx)
    q_seq = np.repeat(np.arange(n_seq), n_q)
    q_pos = rng.integers(0, ctx // repeat, n_seq * n_q)
    q_pos[0], q_pos[-1] = ctx // repeat - 1, ctx + 1000                    # the last token, and a query behind every token
    q = torch.randn(n_seq * n_q, hkv * rep, 128, generator=torch.Generator().manual_seed(ctx)).to(dtype)
    (max_abs, rel_l2), _, _ = _case(B, li, ranks, q, q_seq, q_pos)
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)


def _filled(B, li, ranks, *, out_dtype=torch.float32, sm_scale=None, **cfg):
    """A cache with the layer's tokens, one compress call."""
    n_seq = int(li.seq_ids.max()) + 1
    sizes = dict(max_seqs=n_seq, max_tokens_per_seq=int(np.bincount(li.seq_ids.numpy()).max()), payload_bytes=int((-(-ranks // 64) * 128).sum()))
    gc = GpuCache(B, n_layers=1, n_q_heads=li.n_q_heads, n_kv_heads=li.n_kv_heads, dtype=li.dtype, out_dtype=out_dtype, **{**sizes, **cfg})
    if sm_scale is not None:
        gc.close()
        gc.cfg.sm_scale = sm_scale
        gc.h = B.twkv_cache_create(gc.cfg, gc.pool)
    B.twkv_cache_set_layer_params(gc.h, 0, li.Uinv_k.cuda(), li.Uinv_v.cuda())
    B.twkv_compress(gc.h, 0, li.xt_k.cuda(), li.xt_v.cuda(), li.seq_ids.cuda(), li.positions.cuda(), None,
                    torch.from_numpy(ranks.astype(np.int16)).cuda(), B.TWKV_GATE_FORCED)
    return gc


def _prefill(B, gc, q, q_seq, q_pos, num_splits=0):
    out = torch.full((len(q_seq), q.shape[1], 128), float("nan"), dtype={0: torch.float16, 1: torch.bfloat16, 2: torch.float32}[gc.cfg.out_dtype],
                     device="cuda")
    B.twkv_prefill_attn(gc.h, 0, q.cuda(), q_seq, q_pos, out, num_splits)
    assert B.twkv_cache_status(gc.h) == B.TWKV_OK
    return out.float().cpu().numpy()


def test_tiled_prefill_with_many_items_that_have_no_keys(B):
    # four sequences over two segments, four items per CTA: in the second segment three sequences out of four have no rows, so
    # the CTAs meet such items one after the other, between items with keys
    n_seq, ctx, n_q, hq = 4, 2100, 600, 64
    li = workloads.build_layer(861, n_seq=n_seq, ctx=ctx, n_q_heads=hq, outlier="pct:1", mode="forced", level_probs=(0.05, 0.15, 0.4, 0.4))
    ranks = li.ranks.numpy().astype(np.int64)
    q_seq = np.repeat(np.arange(n_seq), n_q)
    q_pos = np.tile(np.arange(ctx - n_q, ctx), n_seq)
    q = torch.randn(n_seq * n_q, hq, 128, generator=torch.Generator().manual_seed(3)).to(torch.float16)
    gc = _filled(B, li, ranks)
    got = _prefill(B, gc, q, q_seq, q_pos)
    assert np.all(np.isfinite(got))
    pick = np.random.default_rng(4).choice(n_seq * n_q, 40, replace=False)
    max_abs, rel_l2 = attn_errors(got[pick], _oracle_prefill(li, ranks, q[pick], q_seq[pick], q_pos[pick]))
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)
    gc.close()


@pytest.mark.parametrize("hkv,rep,ctx,n_q", [
    (8, 4, 1000, 8),                             # several splits of one segment
    (1, 8, 9000, 33),                            # several segments, then the join of their results
    (2, 4, 100, 50),                             # one split of one segment is the whole result
])
def test_tiled_prefill_shows_a_key_that_is_not_a_number(B, hkv, rep, ctx, n_q):
    # a NaN in one token's key: the queries that see the token get NaN, the others what they would get without it
    bad = ctx // 3
    li = workloads.build_layer(870 + ctx, n_seq=1, ctx=ctx, n_q_heads=hkv * rep, n_kv_heads=hkv, n_calib=256 * hkv, mode="forced", rank_recipe="any")
    ranks = li.ranks.numpy().astype(np.int64)
    q_pos = np.sort(np.random.default_rng(1).integers(0, ctx, n_q))
    q_pos[0], q_pos[1], q_pos[-1] = bad - 1, bad, ctx - 1
    q_seq = np.zeros(n_q, np.int64)
    q = torch.randn(n_q, hkv * rep, 128, generator=torch.Generator().manual_seed(2)).to(torch.float16)
    want = _oracle_prefill(li, ranks, q, q_seq, q_pos)
    li.xt_k[(li.positions == bad).nonzero()[0], 0] = float("nan")
    gc = _filled(B, li, ranks)
    got = _prefill(B, gc, q, q_seq, q_pos)
    gc.close()
    sees = q_pos >= bad
    assert np.all(np.isnan(got[sees]))
    max_abs, rel_l2 = attn_errors(got[~sees], want[~sees])
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)


@pytest.mark.parametrize("hkv,rep,dtype,ctx,n_q,x_scale,u_scale,every", [
    (8, 4, torch.float16, 500, 150, 2.0 ** -13, 1.0, 1),       # values around 1e-4: one f16 low part would keep 12 bits of them
    (8, 4, torch.float16, 500, 8, 2.0 ** 11, 64.0, 37),        # one token in 37 with values around 1e5, beyond f16; several splits
    (3, 2, torch.float16, 300, 100, 2.0 ** 11, 64.0, 2),       # one head per slab
    (1, 8, torch.float16, 9000, 33, 2.0 ** -10, 1.0, 3),       # several segments, large and small values mixed
    (2, 4, torch.bfloat16, 200, 50, 2.0 ** 40, 1.0, 2),        # bf16 states far beyond f16
])
def test_tiled_prefill_values_of_any_size(B, hkv, rep, dtype, ctx, n_q, x_scale, u_scale, every):
    # Rebuilt values are carried as two f16; their size must not cost precision.  fp32 output, so that nothing hides it: keys and
    # weights of 22 bits with scores of a few tens (2^-21 x 20) and the fp32 sums stay below 2e-5, values clamped or without a low
    # part give 1e-4 and more.
    li = workloads.build_layer(880 + ctx, n_seq=1, ctx=ctx, n_q_heads=hkv * rep, n_kv_heads=hkv, n_calib=256 * hkv, dtype=dtype, mode="forced",
                               rank_recipe="any")
    li.xt_v[::every] = (li.xt_v[::every].float() * x_scale).to(dtype)
    li.Uinv_v = (li.Uinv_v.float() * u_scale).to(dtype)
    ranks = li.ranks.numpy().astype(np.int64)
    q_pos = np.sort(np.random.default_rng(1).integers(0, ctx, n_q))
    q_seq = np.zeros(n_q, np.int64)
    q = torch.randn(n_q, hkv * rep, 128, generator=torch.Generator().manual_seed(2)).to(dtype)
    gc = _filled(B, li, ranks)
    got = _prefill(B, gc, q, q_seq, q_pos)
    gc.close()
    _, rel_l2 = attn_errors(got, _oracle_prefill(li, ranks, q, q_seq, q_pos))
    assert rel_l2 < 2e-5, rel_l2


def test_tiled_prefill_shows_an_infinite_value(B):
    li = workloads.build_layer(885, n_seq=1, ctx=300, n_q_heads=32, mode="forced", rank_recipe="any")
    ranks = li.ranks.numpy().astype(np.int64)
    li.xt_v[(li.positions == 200).nonzero()[0], 0] = float("inf")
    gc = _filled(B, li, ranks)
    q_pos = np.arange(100, 300)
    got = _prefill(B, gc, torch.ones(200, 32, 128, dtype=torch.float16), np.zeros(200, np.int64), q_pos)
    gc.close()
    assert not np.isfinite(got[q_pos >= 200]).any()
    assert np.isfinite(got[q_pos < 128]).all()                 # (a block of keys that the token is not in)


@pytest.mark.parametrize("n_q", [6, 300])
def test_tiled_prefill_does_not_depend_on_the_room_in_the_cache(B, n_q):
    # the same chunk in a cache that just holds its sequence, and in one with room for 131072 tokens a sequence and other sequences
    # resident: the same form, splits and bits
    ctx, other = 1000, 30000
    li = workloads.build_layer(891, n_seq=1, ctx=ctx, n_q_heads=32, outlier="pct:1", mode="forced", rank_recipe="any")
    ranks = li.ranks.numpy().astype(np.int64)
    q_pos = np.arange(ctx - n_q, ctx)
    q = torch.randn(n_q, 32, 128, generator=torch.Generator().manual_seed(5)).to(torch.float16)
    gc = _filled(B, li, ranks)
    fitted = _prefill(B, gc, q, np.zeros(n_q, np.int64), q_pos)
    gc.close()
    max_abs, rel_l2 = attn_errors(fitted, _oracle_prefill(li, ranks, q, np.zeros(n_q, np.int64), q_pos))
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)
    li.seq_ids = li.seq_ids + 1
    gc = _filled(B, li, ranks, max_seqs=3, max_tokens_per_seq=131072, payload_bytes=2 * other * 256 + ctx * 4096)
    x = torch.randn(other, 1024, device="cuda").to(torch.float16)
    seq, pos = torch.arange(other, device="cuda", dtype=torch.int32) % 2 * 2, torch.arange(other, device="cuda", dtype=torch.int32) // 2
    B.twkv_compress(gc.h, 0, x, x, seq, pos, None, torch.full((other, 2), 64, dtype=torch.int16, device="cuda"), B.TWKV_GATE_FORCED)
    roomy = _prefill(B, gc, q, np.ones(n_q, np.int64), q_pos)
    assert B.twkv_cache_check(gc.h) == (B.TWKV_OK, 0)
    gc.close()
    np.testing.assert_array_equal(roomy, fitted)


@pytest.mark.parametrize("n_q,repeat", [(33, 64), (200, 30)])
def test_tiled_prefill_of_more_tokens_than_positions(B, n_q, repeat):
    # positions shared by so many tokens that the rows go on past the segments that the positions alone would need
    ctx = 9000
    li = workloads.build_layer(895, n_seq=1, ctx=ctx, n_q_heads=8, n_kv_heads=1, n_calib=256, mode="forced", rank_recipe="any", shuffle_positions=True)
    li.positions = li.positions // repeat
    ranks = li.ranks.numpy().astype(np.int64)
    q_pos = np.random.default_rng(6).integers(0, ctx // repeat, n_q)
    q_pos[0] = ctx // repeat
    q_seq = np.zeros(n_q, np.int64)
    q = torch.randn(n_q, 8, 128, generator=torch.Generator().manual_seed(6)).to(torch.float16)
    gc = _filled(B, li, ranks, max_tokens_per_seq=50000)
    got = _prefill(B, gc, q, q_seq, q_pos)
    gc.close()
    max_abs, rel_l2 = attn_errors(got, _oracle_prefill(li, ranks, q, q_seq, q_pos))
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)


def test_tiled_prefill_is_as_exact_as_decode(B):
    # The last query of a chunk sees what a decode query sees.  Both forms carry keys, weights and values in 22 bits; what differs is
    # how often the tensor core cuts its fp32 sums.  Mean relative error against the oracle: decode 2.4e-6 over six draws; the
    # tiled form had 2.9e-6 with the small products of a block of keys behind the large one.
    n_q, ctx, hq, err = 80, 200, 32, []
    for seed in range(701, 707):
        li = workloads.build_layer(seed, n_seq=2, ctx=ctx, n_q_heads=hq, mode="forced", outlier="pct:1")
        ranks = li.ranks.numpy().astype(np.int64)
        q_seq, q_pos, last = np.repeat([0, 1], n_q), np.tile(np.arange(ctx - n_q, ctx), 2), [n_q - 1, 2 * n_q - 1]
        q = torch.randn(2 * n_q, hq, 128, generator=torch.Generator().manual_seed(9 + seed)).to(torch.float16)
        gc = _filled(B, li, ranks)
        tiled = _prefill(B, gc, q, q_seq, q_pos)[last]
        out = torch.empty(2, hq, 128, device="cuda")
        B.twkv_decode_attn(gc.h, 0, q[last].cuda(), torch.tensor([0, 1], dtype=torch.int32, device="cuda"), out)
        want = _oracle_prefill(li, ranks, q[last], q_seq[last], q_pos[last])
        err.append((attn_errors(tiled, want)[1], attn_errors(out.cpu().numpy(), want)[1]))
        gc.close()
    tiled, decode = np.mean(err, axis=0)
    assert tiled < 1.15 * decode, (tiled, decode)


@pytest.mark.parametrize("n_q", [60, 8])         # one split: written by the attention kernel; several: by the kernel that joins them
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
def test_tiled_prefill_output_types(B, dtype, n_q):
    # a 16-bit output is the fp32 one rounded to nearest even, bit for bit
    ctx = 100 if n_q == 60 else 700
    li = workloads.build_layer(897, n_seq=1, ctx=ctx, n_q_heads=12, n_kv_heads=3, n_calib=768, dtype=dtype, mode="forced", rank_recipe="any")
    ranks = li.ranks.numpy().astype(np.int64)
    q_pos, q_seq = np.arange(ctx - n_q, ctx), np.zeros(n_q, np.int64)
    q = torch.randn(n_q, 12, 128, generator=torch.Generator().manual_seed(7)).to(dtype)
    got = {}
    for od in (torch.float32, torch.float16, torch.bfloat16):
        gc = _filled(B, li, ranks, out_dtype=od)
        got[od] = torch.from_numpy(_prefill(B, gc, q, q_seq, q_pos))
        gc.close()
    max_abs, rel_l2 = attn_errors(got[torch.float32].numpy(), _oracle_prefill(li, ranks, q, q_seq, q_pos))
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)
    for od in (torch.float16, torch.bfloat16):
        torch.testing.assert_close(got[od], got[torch.float32].to(od).float(), rtol=0, atol=0)


@pytest.mark.parametrize("sm_scale", [-0.11, 0.0, 0.5])
def test_tiled_prefill_score_scales(B, sm_scale):
    li = workloads.build_layer(898, n_seq=2, ctx=150, n_q_heads=8, n_kv_heads=2, n_calib=512, mode="forced", rank_recipe="any")
    ranks = li.ranks.numpy().astype(np.int64)
    q_seq, q_pos = np.repeat([0, 1], 40), np.tile(np.arange(110, 150), 2)
    q = torch.randn(80, 8, 128, generator=torch.Generator().manual_seed(8)).to(torch.float16)
    gc = _filled(B, li, ranks, sm_scale=sm_scale)
    got = _prefill(B, gc, q, q_seq, q_pos)
    gc.close()
    scale = float(np.float32(sm_scale))
    w = lambda t: oracle.widen16(bits16(t), "f16")
    want = np.zeros((80, 8, 128))
    for s in (0, 1):
        idx, rows = np.nonzero(li.seq_ids.numpy() == s)[0], q_seq == s
        want[rows] = oracle.prefill_attn(w(li.xt_k)[idx], w(li.xt_v)[idx], ranks[idx, 0], ranks[idx, 1], li.positions.numpy()[idx], w(li.Uinv_k),
                                         w(li.Uinv_v), w(q)[rows], q_pos[rows], 2, 500000.0, scale)
    max_abs, rel_l2 = attn_errors(got, want)
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)


@pytest.mark.parametrize("scale,code", [(1.0, 0), (3000.0, 5)])
def test_tiled_prefill_reports_clamped_keys_when_asked(B, monkeypatch, scale, code):
    # a cache created with TWKV_DEBUG=1 reports rotated keys beyond the f16 range (here up to around 1e5), and only those
    monkeypatch.setenv("TWKV_DEBUG", "1")
    li = workloads.build_layer(899, n_seq=1, ctx=200, n_q_heads=8, n_kv_heads=2, n_calib=512, mode="forced", outlier="none", rank_recipe="any")
    li.xt_k = (li.xt_k.float() * scale).to(torch.float16)
    li.Uinv_k = (li.Uinv_k.float() * min(scale, 10.0)).to(torch.float16)
    ranks = li.ranks.numpy().astype(np.int64)
    gc = _filled(B, li, ranks)
    out = torch.empty(50, 8, 128, device="cuda")
    B.twkv_prefill_attn(gc.h, 0, torch.ones(50, 8, 128, dtype=torch.float16, device="cuda"), np.zeros(50, np.int64), np.arange(150, 200), out)
    assert B.twkv_cache_status(gc.h) == code
    gc.close()


@pytest.mark.parametrize("counts,num_splits", [
    ((3, 1), 0),                                 # three passes, the later ones for one sequence alone
    ((2, 3), 5),                                 # three passes, the splits given by the caller
    ((4, 4), 0),                                 # one query more: the tiled form
])
def test_prefill_on_both_sides_of_the_rule(B, counts, num_splits):
    # few queries per sequence over 2 x 6000 tokens: passes of the decode kernels, one after the other over the same scratch
    ctx, n_q = 6000, sum(counts)
    li = workloads.build_layer(865, n_seq=2, ctx=ctx, n_q_heads=8, n_kv_heads=1, n_calib=256, outlier="pct:1", mode="forced", rank_recipe="any",
                               shuffle_positions=True)
    ranks = li.ranks.numpy().astype(np.int64)
    rng = np.random.default_rng(n_q)
    perm = rng.permutation(n_q)
    q_seq, q_pos = np.repeat([0, 1], counts)[perm], rng.integers(0, ctx, n_q)
    q_pos[[list(q_seq).index(0), list(q_seq).index(1)]] = ctx - 1
    q = torch.randn(n_q, 8, 128, generator=torch.Generator().manual_seed(9)).to(torch.float16)
    gc = _filled(B, li, ranks)
    launches = B.twkv_launch_count()
    got = _prefill(B, gc, q, q_seq, q_pos, num_splits)
    launches = B.twkv_launch_count() - launches
    assert (launches == 4 * max(counts) + 1) == (max(counts) == 3), launches       # four kernels a pass, and the first one's set-up
    assert B.twkv_cache_check(gc.h) == (B.TWKV_OK, 0)
    max_abs, rel_l2 = attn_errors(got, _oracle_prefill(li, ranks, q, q_seq, q_pos))
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)
    if num_splits:
        with pytest.raises(B.TwkvError) as err:                                     # more splits than the partial results have room for
            B.twkv_prefill_attn(gc.h, 0, q.cuda(), q_seq, q_pos, torch.empty(n_q, 8, 128, device="cuda"), 1000)
        assert err.value.code == B.TWKV_ERR_INVALID_ARG
    gc.close()


def test_prefill_of_many_sequences_at_the_last_positions(B):
    # 65 sequences asked for at the last position there is: their bitmaps fill the region they live in, so the call takes several runs
    n_seq, ctx, n_q = 65, 100, 8
    li = workloads.build_layer(866, n_seq=n_seq, ctx=ctx, n_q_heads=8, n_kv_heads=1, n_calib=256, mode="forced", rank_recipe="any")
    ranks = li.ranks.numpy().astype(np.int64)
    q_seq = np.tile(np.arange(n_seq), n_q)
    q_pos = np.full(n_seq * n_q, 524287)
    q_pos[:n_seq], q_pos[n_seq] = 40, 2 ** 31 - 1
    q = torch.randn(n_seq * n_q, 8, 128, generator=torch.Generator().manual_seed(9)).to(torch.float16)
    gc = _filled(B, li, ranks)
    got = _prefill(B, gc, q, q_seq, q_pos)
    gc.close()
    max_abs, rel_l2 = attn_errors(got, _oracle_prefill(li, ranks, q, q_seq, q_pos))
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)


@pytest.mark.parametrize("lengths,n_q", [
    ((9000, 300, 5000, 2000, 4000), 40),         # one alone over two segments, then runs of three and one
    ((130, 70, 9), 3),                           # all in one run
])
def test_prefill_of_sequences_of_different_lengths(B, lengths, n_q):
    # sequences that fit a segment together share a run of the tiled kernels, longer ones have one of their own
    n_seq, ctx = len(lengths), max(lengths)
    li = workloads.build_layer(867, n_seq=n_seq, ctx=ctx, n_q_heads=8, n_kv_heads=1, n_calib=256, mode="forced", rank_recipe="any")
    stay = li.positions < torch.tensor(lengths, dtype=torch.int32)[li.seq_ids.long()]
    for name in ["xt_k", "xt_v", "seq_ids", "positions", "ranks"]:
        setattr(li, name, getattr(li, name)[stay].contiguous())
    ranks = li.ranks.numpy().astype(np.int64)
    rng = np.random.default_rng(10)
    perm = rng.permutation(n_seq * n_q)
    q_seq = np.repeat(np.arange(n_seq), n_q)[perm]
    q_pos = np.concatenate([np.sort(rng.integers(0, n, n_q)) for n in lengths])[perm]
    q = torch.randn(n_seq * n_q, 8, 128, generator=torch.Generator().manual_seed(9)).to(torch.float16)
    gc = _filled(B, li, ranks)
    got = _prefill(B, gc, q, q_seq, q_pos)
    assert B.twkv_cache_check(gc.h) == (B.TWKV_OK, 0)
    gc.close()
    max_abs, rel_l2 = attn_errors(got, _oracle_prefill(li, ranks, q, q_seq, q_pos))
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)


def test_prefill_of_few_queries_over_many_long_sequences_runs_in_passes(B):
    # eight queries each over sixteen sequences that fill a segment of their own: a run of the tiled kernels per sequence would take
    # three times the passes' time
    n_seq, ctx, n_q = 16, 8192, 8
    li = workloads.build_layer(868, n_seq=n_seq, ctx=ctx, n_q_heads=8, n_kv_heads=1, n_calib=256, mode="forced", rank_recipe="any")
    ranks = li.ranks.numpy().astype(np.int64)
    q_seq, q_pos = np.repeat(np.arange(n_seq), n_q), np.tile(np.arange(ctx - n_q, ctx), n_seq)
    q = torch.randn(n_seq * n_q, 8, 128, generator=torch.Generator().manual_seed(9)).to(torch.float16)
    gc = _filled(B, li, ranks)
    launches = B.twkv_launch_count()
    got = _prefill(B, gc, q, q_seq, q_pos)
    assert B.twkv_launch_count() - launches == 4 * n_q + 1
    gc.close()
    pick = np.arange(0, n_seq * n_q, 13)
    max_abs, rel_l2 = attn_errors(got[pick], _oracle_prefill(li, ranks, q[pick], q_seq[pick], q_pos[pick]))
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)


def test_tiled_prefill_where_fewer_rows_exist_than_positions_allow(B):
    # 40 sequences are asked for, 15 hold tokens: planned for two segments by the positions, all rows lie in the first
    n_seq, held, ctx, n_q = 40, 15, 100, 5
    li = workloads.build_layer(869, n_seq=n_seq, ctx=ctx, n_q_heads=4, n_kv_heads=2, n_calib=512, dtype=torch.bfloat16, mode="forced", rank_recipe="any")
    stay = li.seq_ids < held
    for name in ["xt_k", "xt_v", "seq_ids", "positions", "ranks"]:
        setattr(li, name, getattr(li, name)[stay].contiguous())
    ranks = li.ranks.numpy().astype(np.int64)
    q_seq, q_pos = np.repeat(np.arange(n_seq), n_q), np.tile(np.arange(ctx - n_q, ctx), n_seq)
    q = torch.randn(n_seq * n_q, 4, 128, generator=torch.Generator().manual_seed(9)).to(torch.bfloat16)
    gc = _filled(B, li, ranks, max_seqs=n_seq)
    got = _prefill(B, gc, q, q_seq, q_pos)
    gc.close()
    some = q_seq < held
    max_abs, rel_l2 = attn_errors(got[some], _oracle_prefill(li, ranks, q[some], q_seq[some], q_pos[some]))
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)
    assert not got[~some].any()

"""The planner of a decode pass where its split of the work changes: few tiles (the KV heads of a tile dealt out to several
CTAs), head counts that do not divide, unlisted sequences in between, a V tile list longer than one block-wide scan."""
import numpy as np
import pytest
import torch

from paper_2603_04411_b200 import workloads
from tests.helpers import GpuCache, attn_errors, merge_variant, oracle_decode

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hkv,rep,n_seq,ctx,recipe,pick", [
    (8, 4, 1, 1, "any", [0]),                   # one tile: every head a part of its own
    (8, 1, 1, 129, "any", [0]),
    (8, 4, 3, 1000, "levels", [2, 0]),          # around ten items: parts of several heads; sequence 1 not listed
    (8, 2, 9, 600, "any", list(range(9))),      # enough items that they stay whole
    (3, 2, 2, 300, "any", [1, 0]),              # an odd number of KV heads, six classes
    (6, 8, 2, 140, "any", [0, 1]),              # heads split in two, not in four
    (1, 1, 1, 133000, "levels", [0]),           # more than 1024 V tiles in one sequence
])
def test_decode_where_the_work_split_changes(hkv, rep, n_seq, ctx, recipe, pick):
    from paper_2603_04411_b200 import build
    build.build()
    from paper_2603_04411_b200 import binding as B
    d = hkv * 128
    li = workloads.build_layer(820 + ctx, n_seq=n_seq, ctx=ctx, n_q_heads=hkv * rep, n_kv_heads=hkv, n_calib=2 * d, outlier="none",
                               mode="forced", rank_recipe=recipe)
    ranks = np.minimum(li.ranks.numpy().astype(np.int64), d)
    gc = GpuCache(B, n_layers=1, n_q_heads=hkv * rep, n_kv_heads=hkv, dtype=torch.float16, out_dtype=torch.float32, max_seqs=n_seq,
                  max_tokens_per_seq=ctx, payload_bytes=int((-(-ranks // 64) * 128).sum()))
    B.twkv_cache_set_layer_params(gc.h, 0, li.Uinv_k.cuda(), li.Uinv_v.cuda())
    B.twkv_compress(gc.h, 0, li.xt_k.cuda(), li.xt_v.cuda(), li.seq_ids.cuda(), li.positions.cuda(), None,
                    torch.from_numpy(ranks.astype(np.int16)).cuda(), B.TWKV_GATE_FORCED)
    li.q = li.q[pick].contiguous()
    out = torch.full((len(pick), hkv * rep, 128), float("nan"), device="cuda")
    B.twkv_decode_attn(gc.h, 0, li.q.cuda(), torch.tensor(pick, dtype=torch.int32, device="cuda"), out)
    assert B.twkv_cache_status(gc.h) == B.TWKV_OK
    max_abs, rel_l2 = attn_errors(out.cpu().numpy(), oracle_decode(li, ranks, pick))
    gc.close()
    assert max_abs < 2e-3 and rel_l2 < 1e-3, (max_abs, rel_l2)      # the bars of every decode test


@pytest.mark.parametrize("hkv,rep,n_seq,ctx", [
    (8, 8, 13, 40), (1, 8, 33, 40), (1, 4, 35, 30), (4, 4, 47, 20), (8, 4, 23, 30),
])
def test_merge_of_medium_batches(hkv, rep, n_seq, ctx):
    test_decode_where_the_work_split_changes(hkv, rep, n_seq, ctx, "any", list(range(n_seq)))


@pytest.mark.parametrize("hkv,rep,n_seq,ctx", [(8, 4, 9, 60), (8, 1, 10, 40), (8, 8, 3, 60), (2, 8, 20, 30), (1, 2, 3, 50)])
def test_merge_rows_per_cluster(hkv, rep, n_seq, ctx):
    test_decode_where_the_work_split_changes(hkv, rep, n_seq, ctx, "any", list(range(n_seq)))


@pytest.mark.parametrize("rows,hkv,rep,n_seq,ctx", [
    (1, 1, 2, 3, 50),           # 16 spectral components per CTA
    (2, 8, 1, 10, 40),          # two slots
    (4, 8, 4, 5, 60),           # the heads of one slot
    (8, 8, 8, 4, 60),           # eight of them
    (8, 8, 4, 9, 60),           # two slots, one in the last cluster
    (16, 8, 4, 15, 30),         # four slots, three in the last cluster
    (16, 2, 8, 37, 30),         # two slots, one in the last cluster; 32 spectral components
    (16, 8, 1, 70, 20),         # sixteen slots, six in the last cluster
    (32, 8, 8, 15, 40),         # wide: four slots, three in the last cluster
    (32, 4, 4, 59, 20),         # eight slots, three in the last; 64 spectral components
    (32, 1, 8, 117, 20),        # one KV head, 16 spectral components
    (32, 1, 4, 227, 12),
])
def test_every_form_of_the_merge(rows, hkv, rep, n_seq, ctx):
    """The sizes are well inside their form on a device of 148 SMs; the form itself is asked of the library's rule."""
    from paper_2603_04411_b200 import build
    build.build()
    from paper_2603_04411_b200 import binding as B
    fit = B.lib._ZN4twkv14merge_clustersEbi(False, torch.cuda.get_device_properties(0).multi_processor_count)    # twkv::merge_clusters
    assert merge_variant(B, n_seq, hkv, rep, fit) == rows, fit
    test_decode_where_the_work_split_changes(hkv, rep, n_seq, ctx, "any", list(range(n_seq)))


@pytest.mark.parametrize("hkv,single,counts", [
    (8, False, {16: 1, 15: 16, 14: 17, 13: 64, 9: 3}),             # 16 + 16 + 32 + 64 rows fill a tile; class 9 stays by itself
    (8, False, {16: 16, 8: 112, 7: 113, 5: 127, 3: 128, 2: 1, 1: 15}),    # rests that fit exactly, that fit nothing, and a full tile between
    (8, True, {12: 200, 10: 33, 9: 130, 1: 129}),                  # single CTAs; full tiles beside the joint one
    (1, False, {2: 5, 1: 140}),                                    # two classes
    (4, False, {k: 40 for k in range(1, 9)}),                      # every class: three joint tiles
])
def test_joint_tiles_of_partly_full_classes(hkv, single, counts, monkeypatch):
    """Three sequences with these tokens per class (K; V in reverse), one a token longer, one holding the widest class alone; decoded
    in two orders, again after an append, and after an eviction."""
    from paper_2603_04411_b200 import binding as B
    if single:
        monkeypatch.setenv("TWKV_KSCORE_SINGLE", "1")
    d, hq = hkv * 128, hkv * 4
    rng = np.random.default_rng(31 * hkv + len(counts))
    per_class = np.concatenate([rng.integers(64 * c - 63, 64 * c + 1, n) for c, n in counts.items()])
    rk = [rng.permutation(per_class), rng.permutation(np.append(per_class, 64 * max(counts))), np.full(7, 64 * max(counts))]
    n = [len(r) for r in rk]
    room = max(n) + 1
    li = workloads.build_layer(77 + hkv, n_seq=3, ctx=room, n_q_heads=hq, n_kv_heads=hkv, n_calib=2 * d, outlier="none", mode="forced",
                               rank_recipe="any")
    ranks = np.zeros((3, room, 2), dtype=np.int64)
    for s in range(3):
        ranks[s, :n[s], 0], ranks[s, :n[s], 1] = rk[s], rk[s][::-1]
        ranks[s, n[s]] = 1                                          # the token appended later
    ranks = ranks.reshape(-1, 2)
    seq, pos = li.seq_ids.numpy(), li.positions.numpy()
    assert np.array_equal(pos.reshape(3, room), np.tile(np.arange(room), (3, 1)))
    first, then = pos < np.array(n)[seq], pos == np.array(n)[seq]
    gc = GpuCache(B, n_layers=1, n_q_heads=hq, n_kv_heads=hkv, dtype=torch.float16, out_dtype=torch.float32, max_seqs=3, max_tokens_per_seq=room,
                  payload_bytes=room * 12 * d)
    B.twkv_cache_set_layer_params(gc.h, 0, li.Uinv_k.cuda(), li.Uinv_v.cuda())

    def compress(rows):
        t = torch.from_numpy(np.nonzero(rows)[0])
        B.twkv_compress(gc.h, 0, li.xt_k[t].cuda(), li.xt_v[t].cuda(), li.seq_ids[t].cuda(), li.positions[t].cuda(), None,
                        torch.from_numpy(ranks[rows].astype(np.int16)).cuda(), B.TWKV_GATE_FORCED)

    def check(rows, order):
        out = torch.full((len(order), hq, 128), float("nan"), device="cuda")
        B.twkv_decode_attn(gc.h, 0, li.q[order].cuda(), torch.tensor(order, dtype=torch.int32, device="cuda"), out)
        assert B.twkv_cache_status(gc.h) == B.TWKV_OK
        t = torch.from_numpy(np.nonzero(rows)[0])
        part = workloads.LayerInputs(**{**vars(li), "xt_k": li.xt_k[t], "xt_v": li.xt_v[t], "seq_ids": li.seq_ids[t], "positions": li.positions[t],
                                        "q": li.q[order]})
        max_abs, rel_l2 = attn_errors(out.cpu().numpy(), oracle_decode(part, ranks[rows], order))
        assert max_abs < 2e-3 and rel_l2 < 1e-3, (max_abs, rel_l2)  # the bars of every decode test

    compress(first)
    check(first, [0, 1, 2])
    check(first, [2, 0])
    compress(then)
    check(first | then, [1, 2, 0])
    keep = np.sort(rng.permutation(n[0])[:n[0] // 2])
    B.twkv_evict(gc.h, 0, 0, torch.from_numpy(keep.astype(np.int32)).cuda())
    check(((first | then) & (seq > 0)) | ((seq == 0) & np.isin(pos, keep)), [0, 1])
    gc.close()


@pytest.mark.parametrize("counts,single", [
    ({16: 16, 8: 64, 3: 32}, False),         # a pass of its own for the panels above the eighth
    ({8: 30, 2: 17, 1: 33}, False),
    ({12: 1, 11: 15, 9: 16, 4: 70}, True),
])
def test_joint_rows_score_as_in_tiles_of_their_own(counts, single, monkeypatch):
    """The same tokens decoded twice, their K rows in one joint tile and in a full tile per class: the tokens that fill the tiles up score
    so low that their weights are zero, and all weight lies in one V tile, so that the outputs are equal bit for bit if the scores are."""
    from paper_2603_04411_b200 import build
    build.build()
    from paper_2603_04411_b200 import binding as B
    if single:
        monkeypatch.setenv("TWKV_KSCORE_SINGLE", "1")
    heads, d, pos_fill = 8, 1024, 1000
    g = torch.Generator().manual_seed(sum(counts))
    n = sum(counts.values())
    assert sum(-(-c // 16) for c in counts.values()) <= 8
    uinv = torch.linalg.qr(torch.randn(d, d, generator=g))[0].half().contiguous()
    q = torch.randn(heads, 128, generator=g).half()
    classes = torch.tensor([c for c, m in counts.items() for _ in range(m)])[torch.randperm(n, generator=g)]
    x = torch.randn(2, n, d, generator=g).half()
    # a filler of rank r: minus the query, rotated back from the filler's position, projected on the r leading axes
    theta = pos_fill * 500000.0 ** (-torch.arange(64, dtype=torch.float64) / 64)
    lo, hi = q[:, :64].double(), q[:, 64:].double()
    back = torch.cat([lo * theta.cos() + hi * theta.sin(), hi * theta.cos() - lo * theta.sin()], 1)
    fill_x = (-600.0 * (uinv.double() @ back.reshape(d))).half()
    fill_classes = torch.tensor([c for c, m in counts.items() for _ in range(128 - m)])
    for c in counts:
        k = (fill_x[:64 * c].double() @ uinv[:64 * c].double()).reshape(heads, 128)
        assert ((k * back).sum(1) * 128 ** -0.5).max() < -150         # 87 below a sequence's maximum and a weight is less than 2^-126: zero

    def decode(filled):
        m = len(fill_classes) if filled else 0
        xk, xv = torch.cat([x[0], fill_x.expand(m, d)]), torch.cat([x[1], torch.zeros(m, d).half()])
        rk = torch.cat([classes, fill_classes[:m]]) * 64
        rv = torch.cat([torch.full((n,), 320), torch.full((m,), 64)])             # the tokens in a V tile of class 5, the fillers in others
        gc = GpuCache(B, n_layers=1, n_q_heads=heads, n_kv_heads=heads, dtype=torch.float16, out_dtype=torch.float32, max_seqs=1,
                      max_tokens_per_seq=2048, payload_bytes=(n + m) * 4 * d)
        u = uinv.cuda()
        B.twkv_cache_set_layer_params(gc.h, 0, u, u)
        pos = torch.cat([torch.arange(n), torch.full((m,), pos_fill)]).to(torch.int32).cuda()
        B.twkv_compress(gc.h, 0, xk.cuda(), xv.cuda(), torch.zeros(n + m, dtype=torch.int32).cuda(), pos, None,
                        torch.stack([rk, rv], 1).to(torch.int16).cuda(), B.TWKV_GATE_FORCED)
        out = torch.full((1, heads, 128), float("nan"), device="cuda")
        B.twkv_decode_attn(gc.h, 0, q[None].cuda(), torch.zeros(1, dtype=torch.int32, device="cuda"), out, 1)
        assert B.twkv_cache_status(gc.h) == B.TWKV_OK
        gc.close()
        return out.cpu()

    assert torch.equal(decode(False), decode(True))

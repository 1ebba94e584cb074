"""Calls captured into CUDA graphs beside eager calls of the same cache: a captured call has not run, its replays see what the cache
holds then, and nothing it took note of on the host may change what later calls do."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_04411_b200 import workloads
from tests.helpers import GATE_MARGIN_COMPUTE, GpuCache, attn_errors, bits16, check_gate_levels, oracle_decode

pytestmark = pytest.mark.gpu

MAX_ABS, REL_L2 = 2e-3, 1e-3                     # the bars of every attention test


@pytest.fixture(scope="module")
def B():
    from paper_2603_04411_b200 import build
    build.build()
    from paper_2603_04411_b200 import binding
    return binding


def _capture(call):
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    return graph


def test_a_captured_first_call_that_never_runs(B):
    # decode and a large gate call lay out copies of the layer's matrices when they meet them first; captured, they have not done so yet
    n_tok, d = 3500, 256
    li = workloads.build_layer(941, n_seq=1, ctx=n_tok, n_q_heads=8, n_kv_heads=2, n_calib=2 * d, outlier="none", mode="forced")
    gc = GpuCache(B, n_layers=1, n_q_heads=8, n_kv_heads=2, dtype=torch.float16, out_dtype=torch.float32, max_seqs=1, max_tokens_per_seq=n_tok,
                  payload_bytes=n_tok * 4 * d)
    gc.close()
    gc.pool.zero_()                                                        # nothing of an earlier cache in the copies' place
    gc.h = B.twkv_cache_create(gc.cfg, gc.pool)
    W = workloads.gate_params(7, d, torch.float16, n_bumps=64, first_dim=64)
    B.twkv_cache_set_layer_params(gc.h, 0, *[t.cuda().contiguous() for t in (li.Uinv_k, li.Uinv_v, *W)])
    args = [t.cuda() for t in (li.xt_k, li.xt_v, li.seq_ids, li.positions)]
    levels, q = torch.zeros(n_tok, 2, dtype=torch.int16, device="cuda"), li.q.cuda()
    out, sid = torch.zeros(1, 8, 128, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")

    def step():
        B.twkv_compress(gc.h, 0, *args, None, levels, B.TWKV_GATE_COMPUTE)
        B.twkv_decode_attn(gc.h, 0, q, sid, out)

    z = [oracle.gate_logits(oracle.widen16(bits16(x), "f16"), oracle.widen16(bits16(w), "f16"), b.double().numpy())
         for x, w, b in ((li.xt_k, W[0], W[2]), (li.xt_v, W[1], W[3]))]

    def check():
        ranks = levels.cpu().numpy().view(np.uint16).astype(np.int64)
        check_gate_levels(ranks, *z, 0.1, GATE_MARGIN_COMPUTE)
        max_abs, rel_l2 = attn_errors(out.cpu().numpy(), oracle_decode(li, ranks, [0]))
        assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)
        assert B.twkv_cache_status(gc.h) == B.TWKV_OK

    graph = _capture(step)
    step()
    check()
    B.twkv_cache_reset(gc.h)
    levels.zero_()
    graph.replay()
    check()
    gc.close()


def _long_layer(ctx):
    li = workloads.build_layer(942, n_seq=1, ctx=ctx, n_q_heads=8, n_kv_heads=1, n_calib=256, outlier="none", mode="forced", rank_recipe="any")
    ranks = li.ranks.numpy().astype(np.int64)
    gc = GpuCache(B=_binding(), n_layers=1, n_q_heads=8, n_kv_heads=1, dtype=torch.float16, out_dtype=torch.float32, max_seqs=1,
                  max_tokens_per_seq=ctx, payload_bytes=int((-(-ranks // 64) * 128).sum()))
    gc.B.twkv_cache_set_layer_params(gc.h, 0, li.Uinv_k.cuda(), li.Uinv_v.cuda())
    dev = [t.cuda() for t in (li.xt_k, li.xt_v, li.seq_ids, li.positions)] + [torch.from_numpy(ranks.astype(np.int16)).cuda()]

    def append(lo, hi, seq=None):
        gc.B.twkv_compress(gc.h, 0, dev[0][lo:hi], dev[1][lo:hi], dev[2][lo:hi] if seq is None else seq, dev[3][lo:hi], None, dev[4][lo:hi],
                           gc.B.TWKV_GATE_FORCED)
    return gc, li, ranks, append


def _binding():
    from paper_2603_04411_b200 import binding
    return binding


def test_a_decode_call_captured_on_an_empty_cache_splits_as_an_eager_one(B):
    # the usual warm-up: the step is captured before there are tokens, its replays meet a long context
    gc, li, ranks, append = _long_layer(16384)
    q, sid = li.q.cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    out = [torch.zeros(1, 8, 128, device="cuda") for _ in range(2)]
    B.twkv_decode_attn(gc.h, 0, q, sid, out[0])
    graph = _capture(lambda: B.twkv_decode_attn(gc.h, 0, q, sid, out[0]))
    for lo, hi in ((0, 300), (300, 16384)):
        append(lo, hi)
        graph.replay()
        B.twkv_decode_attn(gc.h, 0, q, sid, out[1])
        torch.testing.assert_close(out[0], out[1], rtol=0, atol=0)
    max_abs, rel_l2 = attn_errors(out[0].cpu().numpy(), oracle_decode(li, ranks, [0]))
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)
    assert B.twkv_cache_status(gc.h) == B.TWKV_OK
    gc.close()


def test_decode_depends_on_the_tokens_in_the_cache_alone(B):
    # calls that were refused leave no trace in the rounding of later ones
    gc, li, ranks, append = _long_layer(16384)
    q, sid = li.q.cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    out = [torch.zeros(1, 8, 128, device="cuda") for _ in range(2)]
    for k in range(2):
        B.twkv_cache_reset(gc.h)
        if k:
            for _ in range(4):
                append(0, 8192, torch.full((8192,), 7, dtype=torch.int32, device="cuda"))     # no such sequence
            assert B.twkv_cache_status(gc.h) == B.TWKV_ERR_INVALID_ARG
        append(0, 8192)
        B.twkv_decode_attn(gc.h, 0, q, sid, out[k])
    assert B.twkv_cache_status(gc.h) == B.TWKV_OK
    torch.testing.assert_close(out[1], out[0], rtol=0, atol=0)
    gc.close()


@pytest.mark.parametrize("n_q", [300, 2])        # the tiled form; two decode passes
def test_a_captured_prefill_call_replays_after_its_lists_are_gone(B, n_q):
    # captured with the first tokens in the cache; the host's lists are overwritten and further tokens appended (by a graph as well)
    ctx = 9000
    gc, li, ranks, append = _long_layer(ctx)
    dn = "f16"
    q = torch.randn(n_q, 8, 128, generator=torch.Generator().manual_seed(8)).to(torch.float16)
    q_dev, out = q.cuda(), [torch.zeros(n_q, 8, 128, device="cuda") for _ in range(2)]
    seq, pos = np.zeros(n_q, np.int32), np.arange(ctx - n_q, ctx, dtype=np.int32)
    append(0, 200)
    B.twkv_prefill_attn(gc.h, 0, q_dev, seq, pos, out[1])                  # the layer's one-time set-up
    lists = seq.copy(), pos.copy()
    graph = _capture(lambda: B.twkv_prefill_attn(gc.h, 0, q_dev, *lists, out[0]))
    more = _capture(lambda: append(200, 8500))
    lists[0][:], lists[1][:] = -5, 1 << 30
    scribble = [np.full(3 * n_q, -7, np.int32) for _ in range(200)]         # where the call's own tables may have been
    more.replay()
    append(8500, ctx)
    graph.replay()
    B.twkv_prefill_attn(gc.h, 0, q_dev, seq, pos, out[1])
    torch.testing.assert_close(out[0], out[1], rtol=0, atol=0)
    pick = np.arange(0, n_q, max(1, n_q // 10))
    U = [oracle.widen16(bits16(u), dn) for u in (li.Uinv_k, li.Uinv_v)]
    want = oracle.prefill_attn(oracle.widen16(bits16(li.xt_k), dn), oracle.widen16(bits16(li.xt_v), dn), ranks[:, 0], ranks[:, 1],
                               li.positions.numpy(), *U, oracle.widen16(bits16(q[pick]), dn), pos[pick], 1, 500000.0, 128 ** -0.5)
    max_abs, rel_l2 = attn_errors(out[0].cpu().numpy()[pick], want)
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)
    assert B.twkv_cache_status(gc.h) == B.TWKV_OK and len(scribble) == 200
    gc.close()

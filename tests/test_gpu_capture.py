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

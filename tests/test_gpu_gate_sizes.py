"""The gate of a COMPUTE-mode call at the sizes where its kernels change: below 128 tokens, from 128 to 3072, above; ragged last
token tiles, one to eight KV heads, and a call captured before the gate's weights were laid out."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_04411_b200 import workloads
from tests.helpers import GATE_MARGIN_COMPUTE, GpuCache, bits16, check_gate_levels

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tok,hkv,dtype,capture", [
    (127, 8, torch.float16, False),
    (128, 8, torch.bfloat16, False),            # one token tile
    (257, 1, torch.float16, False),             # one slab of columns a side, one token in the last tile
    (300, 2, torch.float16, True),
    (1500, 3, torch.bfloat16, False),
    (3072, 4, torch.float16, False),            # the largest spread call: more items than SMs
    (3072, 8, torch.bfloat16, False),
    (3073, 8, torch.float16, False),            # the smallest fused ones: CTA pairs, and single CTAs where d_kv / 256 is no whole number
    (3100, 3, torch.bfloat16, False),
])
def test_gate_ranks_where_the_kernels_change(n_tok, hkv, dtype, capture):
    from paper_2603_04411_b200 import build
    build.build()
    from paper_2603_04411_b200 import binding as B
    dn, d = ("f16" if dtype == torch.float16 else "bf16"), hkv * 128
    li = workloads.build_layer(910 + n_tok, n_seq=1, ctx=n_tok, n_q_heads=hkv, n_kv_heads=hkv, n_calib=2 * d, dtype=dtype, outlier="none",
                               mode="forced")
    W = workloads.gate_params(5 + n_tok, d, dtype, n_bumps=min(64, d // 4), first_dim=min(64, d // 4))
    z = [oracle.gate_logits(oracle.widen16(bits16(x), dn), oracle.widen16(bits16(w), dn), b.double().numpy())
         for x, w, b in ((li.xt_k, W[0], W[2]), (li.xt_v, W[1], W[3]))]
    gc = GpuCache(B, n_layers=1, n_q_heads=hkv, n_kv_heads=hkv, dtype=dtype, out_dtype=torch.float32, max_seqs=1,
                  max_tokens_per_seq=n_tok, payload_bytes=n_tok * 4 * d)
    gate = [t.cuda().contiguous() for t in W]
    B.twkv_cache_set_layer_params(gc.h, 0, li.Uinv_k.cuda(), li.Uinv_v.cuda(), *gate)
    args = [t.cuda() for t in (li.xt_k, li.xt_v, li.seq_ids, li.positions)]
    levels = [torch.zeros(n_tok, 2, dtype=torch.int16, device="cuda") for _ in range(2)]
    graph = torch.cuda.CUDAGraph() if capture else None
    if capture:
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            B.twkv_compress(gc.h, 0, *args, None, levels[1], B.TWKV_GATE_COMPUTE)
    B.twkv_compress(gc.h, 0, *args, None, levels[0], B.TWKV_GATE_COMPUTE)      # with a captured one pending: nothing of it has run
    if capture:
        torch.cuda.synchronize()
        B.twkv_cache_reset(gc.h)
        graph.replay()
    for lv in levels[: 1 + capture]:
        n_loose = check_gate_levels(lv.cpu().numpy().view(np.uint16).astype(np.int64), *z, 0.1, GATE_MARGIN_COMPUTE)
        assert n_loose <= 0.05 * 2 * n_tok + 2, n_loose
    assert B.twkv_cache_status(gc.h) == B.TWKV_OK
    gc.close()


def test_gate_ranks_of_a_middle_sized_call_follow_the_weights_as_they_are():
    # weights changed in place between two calls, and a large call captured into a graph that never runs: what a call of 128 to
    # 3072 tokens ranks by are the weights in the caller's memory at that moment
    from paper_2603_04411_b200 import build
    build.build()
    from paper_2603_04411_b200 import binding as B
    n_tok, d, dtype = 300, 256, torch.float16
    li = workloads.build_layer(931, n_seq=1, ctx=4000, n_q_heads=2, n_kv_heads=2, n_calib=2 * d, dtype=dtype, outlier="none", mode="forced")
    gc = GpuCache(B, n_layers=1, n_q_heads=2, n_kv_heads=2, dtype=dtype, out_dtype=torch.float32, max_seqs=1, max_tokens_per_seq=4000,
                  payload_bytes=4000 * 4 * d)
    args = [t.cuda() for t in (li.xt_k, li.xt_v, li.seq_ids, li.positions)]
    gate = [t.cuda().contiguous() for t in workloads.gate_params(5, d, dtype, n_bumps=64, first_dim=64)]
    B.twkv_cache_set_layer_params(gc.h, 0, li.Uinv_k.cuda(), li.Uinv_v.cuda(), *gate)
    levels = torch.zeros(4000, 2, dtype=torch.int16, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.twkv_compress(gc.h, 0, *args, None, levels, B.TWKV_GATE_COMPUTE)
    for seed in (5, 6):
        W = workloads.gate_params(seed, d, dtype, n_bumps=64, first_dim=64)
        for have, new in zip(gate, W):
            have.copy_(new)
        B.twkv_cache_reset(gc.h)
        B.twkv_compress(gc.h, 0, *[t[:n_tok] for t in args], None, levels, B.TWKV_GATE_COMPUTE)
        z = [oracle.gate_logits(oracle.widen16(bits16(x[:n_tok]), "f16"), oracle.widen16(bits16(w), "f16"), b.double().numpy())
             for x, w, b in ((li.xt_k, W[0], W[2]), (li.xt_v, W[1], W[3]))]
        check_gate_levels(levels[:n_tok].cpu().numpy().view(np.uint16).astype(np.int64), *z, 0.1, GATE_MARGIN_COMPUTE)
    assert B.twkv_cache_status(gc.h) == B.TWKV_OK
    gc.close()

"""Compress calls of at most 128 tokens (one kernel for ranks, allocation and rows), the cache image bit for bit."""
import numpy as np
import pytest
import torch

from paper_2603_04411_b200 import workloads
from tests.test_gpu_parity import GATE_MARGIN_LOGITS, B, MAX_ABS, REL_L2, run_case, settle_logits, to_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hkv,n_seq,classes,sizes", [
    (8, 3, 16, [128, 1, 127, 33, 16, 128, 31]),        # many keys, every remainder of a warp
    (8, 1, 1, [128, 1, 127, 128]),                     # one key: a full tile, a new one, its rest
    (3, 5, 6, [32, 64, 97, 2]),                        # 384 components
    (1, 64, 2, [64, 128, 64]),                         # a token per sequence
])
def test_small_calls_place_their_rows(B, hkv, n_seq, classes, sizes):  # noqa: F811
    n = sum(sizes)
    ctx = -(-n // n_seq)
    li = workloads.build_layer(5 + hkv, n_seq=n_seq, ctx=ctx, n_q_heads=2 * hkv, n_kv_heads=hkv, n_calib=256 * hkv, outlier="none", mode="forced",
                               rank_recipe="any")
    order = torch.argsort(li.positions, stable=True)[:n]                   # a step of every sequence after the other
    for name in ["xt_k", "xt_v", "seq_ids", "positions"]:
        setattr(li, name, getattr(li, name)[order].contiguous())
    ranks = np.random.default_rng(n).integers(1, 64 * classes + 1, (n, 2)).astype(np.int64)
    ends = np.cumsum(sizes)
    calls = [(int(e - s), int(e)) for s, e in zip(sizes, ends)]
    (max_abs, rel_l2), _, _ = run_case(B, to_cuda(li), ranks, mode=B.TWKV_GATE_FORCED, calls=calls, max_tokens_per_seq=ctx)
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)


@pytest.mark.parametrize("n_tok", [1, 16, 127, 128])
def test_small_calls_rank_their_logits(B, n_tok):  # noqa: F811
    li = workloads.build_layer(40, n_seq=1, ctx=n_tok, n_q_heads=8, n_calib=2048, outlier="none", mode="logits")
    ranks, _ = settle_logits(li.logits, 0.1, GATE_MARGIN_LOGITS)
    (max_abs, rel_l2), _, _ = run_case(B, to_cuda(li), ranks.astype(np.int64), mode=B.TWKV_GATE_LOGITS)
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)

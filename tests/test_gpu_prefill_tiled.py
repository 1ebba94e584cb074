"""The tiled form of chunked-prefill attention where its work split changes, against the CPU oracle: several segments of rows,
several groups of query blocks, an odd number of KV heads, repeated positions, a block of one tile beside a block of two.
Bars as for every attention test (max-abs 2e-3, relative L2 1e-3)."""
import numpy as np
import pytest
import torch

from paper_2603_04411_b200 import workloads
from tests.test_gpu_prefill import MAX_ABS, REL_L2, B, _case

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

"""Compress calls of at most 128 tokens, the cache image bit for bit: up to 32 tokens one kernel ranks, allocates and moves the rows,
beyond that the allocation and the rows (and, with logits, the ranks) have kernels of their own."""
import numpy as np
import pytest
import torch

from oracle.cache_image import CacheImage
from paper_2603_04411_b200 import workloads
from tests.helpers import GpuCache, bits16, compare_cache_with_image
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


@pytest.mark.parametrize("n_tok", [1, 16, 31, 32, 33, 127, 128])
def test_small_calls_rank_their_logits(B, n_tok):  # noqa: F811
    li = workloads.build_layer(40, n_seq=1, ctx=n_tok, n_q_heads=8, n_calib=2048, outlier="none", mode="logits")
    ranks, _ = settle_logits(li.logits, 0.1, GATE_MARGIN_LOGITS)
    (max_abs, rel_l2), _, _ = run_case(B, to_cuda(li), ranks.astype(np.int64), mode=B.TWKV_GATE_LOGITS)
    assert max_abs < MAX_ABS and rel_l2 < REL_L2, (max_abs, rel_l2)


class _Appends:
    """A cache whose blocks start as 0xff bytes and its image, compared after every call."""

    def __init__(self, B, n_seq, room, hkv=8):  # noqa: F811
        self.B, self.d = B, 128 * hkv
        self.gc = GpuCache(B, n_layers=1, n_q_heads=2 * hkv, n_kv_heads=hkv, dtype=torch.float16, out_dtype=torch.float32, max_seqs=n_seq,
                           max_tokens_per_seq=room, payload_bytes=n_seq * room * 4 * self.d)
        self.gc.pool[int(self.gc.lay.blocks_off):] = 0xFF
        self.img = CacheImage(1, self.d, n_seq, room, int(self.gc.lay.n_blocks))
        self.g = torch.Generator().manual_seed(97 * n_seq + room)
        self.have = [0] * n_seq

    def call(self, seqs, ranks, refused=None):
        """Appends a token to every sequence of `seqs`, in that order; `refused`: the status the call has to end with."""
        B, n = self.B, len(seqs)  # noqa: F811
        pos, have = np.zeros(n, dtype=np.int32), list(self.have)
        for i, s in enumerate(seqs):
            pos[i] = have[s]
            have[s] += 1
        x = torch.randn(2, n, self.d, generator=self.g).half()
        ranks = np.asarray(ranks, dtype=np.int64)
        B.twkv_compress(self.gc.h, 0, x[0].cuda(), x[1].cuda(), torch.tensor(seqs, dtype=torch.int32).cuda(), torch.from_numpy(pos).cuda(), None,
                        torch.from_numpy(ranks.astype(np.int16)).cuda(), B.TWKV_GATE_FORCED)
        assert B.twkv_cache_status(self.gc.h) == (B.TWKV_OK if refused is None else refused)
        if refused is None:
            assert self.img.append(0, bits16(x[0]), bits16(x[1]), np.array(seqs), pos, ranks)
            self.have = have
        compare_cache_with_image(self.gc, self.img)

    def close(self):
        assert self.B.twkv_cache_check(self.gc.h, -1) == (self.B.TWKV_OK, 0)
        self.gc.close()


@pytest.mark.parametrize("sizes", [
    [8, 32, 33], [1, 31, 1],             # into an empty key, then behind it
    [125, 8], [127, 32], [120, 33],      # the rest of a tile and the start of the next one
    [125, 3, 2], [96, 32, 32],           # exactly full, then a new tile
    [128, 32], [128, 128, 1],            # behind a full tile
])
def test_tokens_of_one_key_around_a_tile(B, sizes):  # noqa: F811
    """Every token of one sequence, K in one class and V in another, ranks at both ends of theirs."""
    a = _Appends(B, 1, sum(sizes))
    rng = np.random.default_rng(sum(sizes))
    for n in sizes:
        a.call([0] * n, np.stack([rng.integers(129, 193, n), np.where(np.arange(n) % 2, 704, 641)], axis=1))
    a.close()


@pytest.mark.parametrize("hkv,n_seq", [(8, 3), (3, 5), (1, 2)])
def test_tokens_that_share_keys(B, hkv, n_seq):  # noqa: F811
    """Calls of a few tokens with two classes per side: several tokens of a key in one call, in any order, over more than a tile."""
    a = _Appends(B, n_seq, 400, hkv)
    rng = np.random.default_rng(hkv)
    for n in [2, 32, 9, 33, 3, 31, 32, 5, 100, 11, 32, 7, 15, 128, 32, 4, 12]:
        a.call(rng.integers(0, n_seq, n).tolist(), rng.choice([1, 64, 65, 128], (n, 2)))
    a.close()


@pytest.mark.parametrize("n", [1, 8, 32, 33, 40])
def test_refused_small_calls_leave_the_tables_alone(B, n):  # noqa: F811
    a = _Appends(B, 2, 90)
    both = [i % 2 for i in range(n)]
    ranks = np.full((n, 2), 300)
    a.call(both, ranks)
    bad = ranks.copy()
    bad[n // 2, 1] = 0                                               # no rank
    a.call(both, bad, refused=B.TWKV_ERR_INVALID_ARG)
    bad[n // 2, 1] = a.d + 1
    a.call(both, bad, refused=B.TWKV_ERR_INVALID_ARG)
    rest = 90 - a.have[1]
    a.call([1] * rest, np.full((rest, 2), 65))
    a.call([1] * n, ranks, refused=B.TWKV_ERR_CAPACITY)               # sequence 1 is full; sequence 0 goes on
    a.call([0] * min(n, 90 - a.have[0]), ranks[:min(n, 90 - a.have[0])])
    a.close()


@pytest.mark.parametrize("n_tok,launches", [(1, (1, 1, 2)), (32, (1, 1, 2)), (33, (2, 3, 4)), (128, (2, 3, 4))])
def test_launches_of_a_small_call(B, n_tok, launches):  # noqa: F811
    """Where the line between the two forms lies: launches with ranks, with logits, and with the gate."""
    d = 1024
    gc = GpuCache(B, n_layers=1, n_q_heads=16, n_kv_heads=8, dtype=torch.float16, out_dtype=torch.float32, max_seqs=1, max_tokens_per_seq=3 * n_tok,
                  payload_bytes=3 * n_tok * 4 * d)
    u = torch.eye(d).half().cuda()
    gate = [t.cuda() for t in workloads.gate_params(3, d, torch.float16)]
    B.twkv_cache_set_layer_params(gc.h, 0, u, u, *gate)
    x, z = torch.randn(n_tok, d).half().cuda(), torch.randn(n_tok, 2, d).cuda()
    seq, levels = torch.zeros(n_tok, dtype=torch.int32, device="cuda"), torch.full((n_tok, 2), 100, dtype=torch.int16, device="cuda")
    for k, (mode, want) in enumerate(zip([B.TWKV_GATE_FORCED, B.TWKV_GATE_LOGITS, B.TWKV_GATE_COMPUTE], launches)):
        pos = torch.arange(k * n_tok, (k + 1) * n_tok, dtype=torch.int32, device="cuda")
        before = B.twkv_launch_count()
        B.twkv_compress(gc.h, 0, x, x, seq, pos, z if mode == B.TWKV_GATE_LOGITS else None, levels, mode)
        assert B.twkv_launch_count() - before == want, (mode, n_tok)
    assert B.twkv_cache_status(gc.h) == B.TWKV_OK
    gc.close()

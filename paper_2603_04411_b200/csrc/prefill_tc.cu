// Chunked-prefill attention on the 5th-generation tensor cores: many causal queries per sequence over the mixed-rank cache.
//
// A decode pass rebuilds every key for one query per sequence; with a chunk of queries that work is shared.  The visible
// tokens of the call's sequences are laid out as dense rows in position order (a sequence starts on a multiple of 128
// rows), and the rows are taken in segments that fit the gate scratch.  Per segment:
//   pf_recon_kernel  rebuilds K^ = X^_K U_K^-1 (rotated by position) and V^ = X^_V U_V^-1 (Eq. 3) once per token into the
//                    segment buffer [KV head][K high | K low | V high | V low][row][128], every value as two 16-bit parts
//   pf_attn_kernel   softmax attention of every block of queries over the segment's rows
// and pf_combine_kernel joins the partial results of the splits at the end.  The tables behind it:
//   pf_init / pf_bits / pf_scan / pf_rows: position bitmap of every sequence's visible tokens -> rank of a position = dense
//   row; per query the number of rows it may see.  Should two visible tokens of a sequence share a position, the rows of that
//   sequence follow the K tiles instead and the causal mask compares positions.
//
// Precision: as in decode attention, keys are carried as two f16 (22 bits) and queries as f16; softmax weights and values are two
// f16 as well, whatever the cache type, so that the result is the spectral-space one to rounding.  The products high.low,
// low.high and high.high of weights and values are formed.
// Rebuilt values may lie outside f16 although the stored 16-bit components do not, or be so small that the low parts lose bits.  A
// few sampled tokens tell the size of the call's values; one power of two brings it near 1 and goes back onto the outputs.  A row
// (token, KV head) whose largest value still lies outside is divided by a power of its own, which its softmax weights carry; blocks of
// keys without such a row (nearly all) run as if there were none.
//
// Cost per 128 x 128 tile of (query row, token): 2 + 3 tensor-core units of 2 x 128^3 flop; the softmax of one tile runs
// beside the products of the other.
#include <type_traits>

#include "twkv_dev.h"
#include "tc_util.cuh"
#include "mma_util.cuh"
#include "scan_util.cuh"
#include "prefill.h"

namespace twkv {
using namespace tc;

// ------------------------------------------------------------------------------------------ tables
// Zeroes the position bitmaps and maps sequence ids to the call's sequence slots.
__global__ void __launch_bounds__(1024) pf_init_kernel(DevView v, PfCall a) {
  chain_start();
  chain_wait();
  for (int i = blockIdx.x * 1024 + threadIdx.x; i < a.n_words; i += gridDim.x * 1024) a.bits[i] = 0u;
  if (blockIdx.x > 0) return;
  for (int s = threadIdx.x; s < v.S; s += 1024) a.slot[s] = -1;
  __syncthreads();
  for (int u = threadIdx.x; u < a.n_u; u += 1024) { a.slot[a.seqs[3 * u]] = u; a.dup[u] = 0; }
  for (int i = threadIdx.x; i < a.seg_rows / TILE * v.Hkv; i += 1024) a.vflag[i] = 0;
  if (threadIdx.x == 0) *a.ticket = 0;
}

// Sets the bit of every visible token's position; a position met twice marks its sequence.
__global__ void __launch_bounds__(1024) pf_bits_kernel(DevView v, PfCall a, int layer) {
  chain_start();
  chain_wait();
  const int sub = threadIdx.x >> 7, slot = threadIdx.x & (TILE - 1);
  const int n = v.ntiles(layer)[0];
  const int4* desc = v.desc(layer, 0);
  const int* kpos = v.aux(layer, 0);
  for (int t = blockIdx.x * 8 + sub; t < n; t += gridDim.x * 8) {
    const int4 d = desc[t];
    const int u = a.slot[d.x];
    if (u < 0 || slot >= d.z) continue;
    const int pos = kpos[(size_t)t * TILE + slot];
    if (pos > a.seqs[3 * u + 1]) continue;
    const unsigned bit = 1u << (pos & 31);
    if (atomicOr(&a.bits[a.seqs[3 * u + 2] + (pos >> 5)], bit) & bit) a.dup[u] = 1;
  }
}

// One CTA per sequence: exclusive prefix of the bitmap's word counts and the number of rows; the last CTA to finish lays
// the sequences out one behind the other.
__global__ void __launch_bounds__(1024) pf_scan_kernel(DevView v, PfCall a, int layer) {
  chain_start();
  chain_wait();
  __shared__ int s_warp[32];
  __shared__ int s_last;
  const int u = blockIdx.x, tid = threadIdx.x;
  const int words = (a.seqs[3 * u + 1] + 32) >> 5, off = a.seqs[3 * u + 2];
  int base = 0;
  for (int w0 = 0; w0 < words; w0 += 1024) {
    const int w = w0 + tid;
    const int c = w < words ? __popc(a.bits[off + w]) : 0;
    int total;
    const int e = block_scan_excl(c, s_warp, &total);
    if (w < words) a.pref[off + w] = base + e;
    base += total;
  }
  if (a.dup[u]) {
    // two tokens on one position: rows in K tile order
    const int seq = a.seqs[3 * u], n = v.ntiles(layer)[0];
    const int4* desc = v.desc(layer, 0);
    base = 0;
    for (int t0 = 0; t0 < n; t0 += 1024) {
      const int t = t0 + tid;
      int c = 0;
      if (t < n) { const int4 d = desc[t]; c = d.x == seq ? d.z : 0; }
      int total;
      const int e = block_scan_excl(c, s_warp, &total);
      for (int s = 0; s < c; ++s) a.krow[(size_t)t * TILE + s] = base + e + s;
      base += total;
    }
  }
  if (tid == 0) {
    a.rows[u] = base;
    __threadfence();
    s_last = atomicAdd(a.ticket, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  int run = 0;
  for (int u0 = 0; u0 < a.n_u; u0 += 1024) {
    const int i = u0 + tid;
    const int r = i < a.n_u ? (*(volatile int*)&a.rows[i] + TILE - 1) / TILE * TILE : 0;
    int total;
    const int e = block_scan_excl(r, s_warp, &total);
    if (i < a.n_u) a.base[i] = run + e;
    run += total;
  }
  if (tid == 0) *a.total = run;
}

// Segments that only repeated positions could reach have been launched as well (their set-up ran beside the kernel before).  Where the
// first segment may be the whole result, a later one without rows must leave too: it would write its nothing over the outputs.
__device__ __forceinline__ bool pf_idle(const PfCall& a, int seg) {
  return seg > 0 && (seg >= a.seg_rest || a.n_splits == 1) && (long long)seg * a.seg_rows >= *a.total;
}
// Whether the attention kernel's result for a query is whole: one split of the only segment with rows.
__device__ __forceinline__ bool pf_whole(const PfCall& a) { return a.n_splits == 1 && *a.total <= a.seg_rows; }

__device__ __forceinline__ int pf_rank(const PfCall& a, int off, int pos) {      // visible tokens before position pos
  const int w = off + (pos >> 5);
  return a.pref[w] + __popc(a.bits[w] & ((1u << (pos & 31)) - 1u));
}

// Size of the call's values: the largest of eight tokens' values, rebuilt from the first 16 components, in one KV head each (a fraction of
// the real ones).  Values near 1 stay as they are; others are brought there by a power of two.  One chain of dependent reads, about as
// long as the other CTAs'.
constexpr int PF_SAMPLE = 16;
template <bool BF16>
__device__ __forceinline__ float pf_sample_value(const uint4* x, const unsigned short* u, int d_kv) {
  unsigned short uj[PF_SAMPLE];
#pragma unroll
  for (int j = 0; j < PF_SAMPLE; ++j) uj[j] = u[(size_t)j * d_kv];
  const uint4 x0 = x[0], x1 = x[1];
  const unsigned w[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
  float sum = 0.f;
#pragma unroll
  for (int j = 0; j < PF_SAMPLE; ++j) sum += to_f32<BF16>((unsigned short)(w[j >> 1] >> (16 * (j & 1)))) * to_f32<BF16>(uj[j]);
  return fabsf(sum);
}
__device__ void pf_value_scale(const DevView& v, const PfCall& a, int layer) {
  __shared__ float s_max[32];
  const int tid = threadIdx.x, k = tid >> 7;
  const int seq = a.seqs[3 * (k * a.n_u / 8)], n = v.svc(layer)[seq];
  float top = 0.f;
  if (n > 0) {
    const int4 d = v.desc(layer, 1)[v.svt(layer)[(size_t)seq * v.TPS + (2 * k + 1) * n / 16]];
    const uint4* x = reinterpret_cast<const uint4*>(v.blocks + (size_t)d.w * BLOCK_BYTES + (d.z >> 1) * (PANEL * 2));
    const unsigned short* u = a.uv + (k % v.Hkv) * HEAD_DIM + (tid & (HEAD_DIM - 1));
    top = v.dtype == TWKV_BF16 ? pf_sample_value<true>(x, u, v.d_kv) : pf_sample_value<false>(x, u, v.d_kv);
  }
  for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
  if ((tid & 31) == 0) s_max[tid >> 5] = top;
  __syncthreads();
  if (tid >= 32) return;
  top = s_max[tid];
  for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
  if (tid > 0) return;
  int e = 0;
  if ((top > 1024.f && top < INFINITY) || (top < 0.0625f && top > 0.f)) e = max((int)(__float_as_uint(top) >> 23) - 127, PF_SCALE_MIN);
  a.vscale[0] = __uint_as_float((unsigned)(127 - min(e, 126)) << 23);
  a.vscale[1] = __uint_as_float((unsigned)(127 + min(e, 126)) << 23);
}

// Dense row of every K and V slot, position of every row, the segments a tile touches; per query and per block of queries
// what it may see.  The last CTA looks at the size of the values, the `qctas` before it take the queries.
__global__ void __launch_bounds__(1024) pf_rows_kernel(DevView v, PfCall a, int layer, int qctas) {
  chain_start();
  chain_wait();
  const int tctas = (int)gridDim.x - 1 - qctas;
  if ((int)blockIdx.x == tctas + qctas) {
    pf_value_scale(v, a, layer);
    return;
  }
  if ((int)blockIdx.x >= tctas) {
    for (int b = ((int)blockIdx.x - tctas) * 32 + (threadIdx.x >> 5); b < a.n_blocks; b += qctas * 32) {       // a warp per block
      const int2 q = a.blocks[b];
      const int u = q.y >> 9, cnt = q.y & 0x1ff, lane = threadIdx.x & 31;
      const int dup = a.dup[u], off = a.seqs[3 * u + 2], maxq = a.seqs[3 * u + 1], R = a.rows[u];
      int most = 0;
      for (int i = lane; i < cnt; i += 32) {
        const int pos = a.qpos[q.x + i];
        // (a position at or past the largest bitmap entry sees every row; the word of pos + 1 may lie outside the bitmap)
        const int vis = dup || pos >= maxq ? R : pf_rank(a, off, pos + 1);
        a.qvis[q.x + i] = vis;
        most = max(most, vis);
      }
      for (int o = 16; o > 0; o >>= 1) most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
      if (lane == 0) a.binfo[b] = make_int4(a.base[u], most, dup, 0);
    }
    return;
  }
  __shared__ int s_lo[32], s_hi[32];
  const int sub = threadIdx.x >> 7, slot = threadIdx.x & (TILE - 1), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nk = v.ntiles(layer)[0], n = nk + v.ntiles(layer)[1];
  const int* kpos = v.aux(layer, 0);
  const int* link = v.aux(layer, 1);
  for (int i = blockIdx.x * 8 + sub; i < n; i += tctas * 8) {
    const int side = i >= nk, t = side ? i - nk : i;
    const int4 d = v.desc(layer, side)[t];
    const int u = a.slot[d.x];
    int row = -1;
    if (u >= 0 && slot < d.z) {
      const int ks = side ? link[(size_t)t * TILE + slot] : t * TILE + slot;
      const int pos = kpos[ks];
      // a sequence with a repeated position keeps every token (rows in K tile order, written by pf_scan)
      if (a.dup[u]) row = a.base[u] + a.krow[ks];
      else if (pos <= a.seqs[3 * u + 1]) row = a.base[u] + pf_rank(a, a.seqs[3 * u + 2], pos);
      if (!side && row >= 0) a.rowpos[row] = pos;
    }
    // a.krow still holds the K-tile-order rows of marked sequences that V slots read, so the K rows go to a table of their own
    (side ? a.vrow : a.krow_out)[(size_t)t * TILE + slot] = row;
    int lo = row >= 0 ? row : 0x7fffffff, hi = row;
    for (int o = 16; o > 0; o >>= 1) {
      lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) { s_lo[warp] = lo; s_hi[warp] = hi; }
    named_bar_sync(1 + sub, TILE);
    if (slot == 0) {
      for (int w = 1; w < 4; ++w) { lo = min(lo, s_lo[warp + w]); hi = max(hi, s_hi[warp + w]); }
      // .z: first and last segment the tile has rows in (first > last: none)
      const int seg = hi >= 0 ? (lo / a.seg_rows) | ((hi / a.seg_rows) << 16) : 1;
      (side ? v.kpairs : v.klist)[t] = make_int4(d.y | (d.z << 8), d.w, seg, 0);
    }
    named_bar_sync(1 + sub, TILE);
  }
}

// ------------------------------------------------------------------------------------------ reconstruction
constexpr int PR_THREADS = 384;                                 // warps 0 and 1: producer and issuer, 4 to 11: epilogue
constexpr int PR_REGS_LIGHT = 56, PR_REGS_EPI = 224;            // 384 threads of 168 registers, divided again by warpgroup
constexpr int PR_STAGES = 3;
constexpr uint32_t PR_A_BYTES = 16384;                          // [128 tokens][64 components]
constexpr uint32_t PR_ATOM_BYTES = 8192;                        // [64 components][64 output dims]: one MN-major atom of U^-1
constexpr uint32_t PR_STAGE_BYTES = PR_A_BYTES + 4 * PR_ATOM_BYTES;
constexpr uint32_t PR_OUT_BYTES = 8192;                         // per warp: 32 half rows of 128 bytes on their way out, both parts
constexpr int PR_ROPE_STRIDE = 33;                              // float4 per row of the small RoPE table (32 + 1 against bank conflicts)
constexpr uint32_t PR_ROPE_BYTES = ROPE_LO * PR_ROPE_STRIDE * 16;
constexpr uint32_t PR_SMEM = PR_STAGES * PR_STAGE_BYTES + 8 * PR_OUT_BYTES + PR_ROPE_BYTES + 8 * (2 * PR_STAGES + 4) + 16;
static_assert(PR_SMEM > CHAIN_TMEM_SMEM, "no other CTA with tensor memory beside this one");
// A row whose largest value (beside the call's scale) lies outside these is scaled by itself: a small one to [2^-3, 2^-2), a large one to
// [2^14, 2^15).  A part is exact to 2^-25, 2^-22 of values of the usual size.  Scaled further up, a small row's weights (which shrink
// by as much) would lose bits beside those of rows that are not scaled.
constexpr float PR_V_MIN = 0x1p-8f, PR_V_MAX = 65504.f;
constexpr int PR_EXP_MIN = -60, PR_EXP_MAX = 113;               // 2^-e times a sum of weights stays an fp32 number
// Panels summed into one accumulator; the sums of several accumulators are added in fp32 registers.  The tensor core cuts its
// fp32 sum after every instruction (K = 16), so the error grows with the length of a chain.  K: eight panels, the length of
// decode attention's passes, so that both round alike.  V: two panels; decode attention sums values over tokens, not over
// components (largest difference between the two at rank 512: 2.9e-6 with eight panels, 1.9e-6 with two).
__host__ __device__ constexpr int pr_chain(int side) { return side ? 2 : 8; }

__device__ __forceinline__ uint64_t pk2(float a, float b) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ uint64_t pk2u(uint32_t a, uint32_t b) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b)); return r; }
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) { uint64_t r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) { uint64_t r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) { uint64_t r; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) { uint64_t r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ float max_abs3(float a, uint32_t b, uint32_t c) {      // the largest magnitude
  float r;
  asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "r"(b), "r"(c));
  return r;
}
__device__ __forceinline__ void unpk2(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
// One work item = (tile, slab of NS = 256 output dims, i.e. two KV heads; 128 where d_kv is not a multiple of 256).
// [128 x NS] accumulators alternate between two TMEM buffers; state panels (K-major A) and U^-1 atoms (rows of the caller's
// matrix as they lie: MN-major B) stream through a ring of three stages.  Eight epilogue warps (thread = one token row x
// half of a head's dims) rotate (K), split into two parts and hand the rows out through shared memory: a row's place in the
// segment buffer is its token's dense row, so a warp stores four whole 128-byte pieces per instruction instead of 32
// scattered 16-byte ones.
// What bounds it: the epilogue's latencies, with two warps per scheduler, and the way of 128 KiB per item into L2 (about 5 TB/s over
// all SMs: the same item takes 3.8 us with 128 live rows and 2.1 with twenty).  So the tables of the next item are read an item ahead,
// a slab is read from tensor memory while the piece before it is rotated, and a part's rows are all read back before the first is
// stored: the segments of 32768 tokens 243 -> 227 us by themselves, five ragged prompts 49 -> 45 (the calls 880 -> 864 and 182 -> 178).
// Storing 32 bytes per thread straight from registers instead is as fast for tiles with few rows and 1.6 times slower for full ones.
template <bool BF16>
__global__ void __launch_bounds__(PR_THREADS, 1)
pf_recon_kernel(const __grid_constant__ CUtensorMap map_blocks, const __grid_constant__ CUtensorMap map_uk,
                const __grid_constant__ CUtensorMap map_uv, DevView v, PfCall a, int layer, int seg) {
  chain_start();
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t s0 = smem_addr(smem_raw);
  unsigned char* out_stage = smem_raw + PR_STAGES * PR_STAGE_BYTES;
  float4* sRope = reinterpret_cast<float4*>(out_stage + 8 * PR_OUT_BYTES);
  unsigned char* tail = out_stage + 8 * PR_OUT_BYTES + PR_ROPE_BYTES;
  const uint32_t bars = smem_addr(tail);
  const uint32_t full = bars, empty = full + 8 * PR_STAGES, acc_full = empty + 8 * PR_STAGES, acc_empty = acc_full + 16;
  uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(tail + 8 * (2 * PR_STAGES + 4));
  volatile int* abort_flag = reinterpret_cast<int*>(s_tmem_base + 1);
  const bool misaligned = (s0 & 1023u) != 0;

  if (tid == 0) {
    for (int i = 0; i < PR_STAGES; ++i) { mbar_init(full + 8 * i, 1); mbar_init(empty + 8 * i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(acc_full + 8 * i, 1); mbar_init(acc_empty + 8 * i, 8); }
    *abort_flag = misaligned ? 1 : 0;
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc(smem_addr(s_tmem_base), 512);
  chain_wait();
  const bool idle = pf_idle(a, seg);
  for (int i = tid; i < ROPE_LO * 32; i += PR_THREADS) sRope[(i >> 5) * PR_ROPE_STRIDE + (i & 31)] = v.rope_lo[i];
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem_base = *s_tmem_base;

  const int NS = v.d_kv % 256 == 0 ? 256 : 128, n_slabs = v.d_kv / NS;
  const int nk = v.ntiles(layer)[0], n_items = (nk + v.ntiles(layer)[1]) * n_slabs;
  const int step = gridDim.x;
  // the items of this CTA whose tile has rows in the segment; every role walks them in the same order, 32 looked up at once
  auto entry = [&](int i, int& side, int& t) -> int4 {
    const int e = i / n_slabs;
    side = e >= nk;
    t = side ? e - nk : e;
    return side ? v.kpairs[t] : v.klist[t];
  };
  auto lookup = [&](int i0) -> unsigned {
    const int i = i0 + lane * step;
    bool mine = false;
    if (i < n_items) {
      int side, t;
      const int z = entry(i, side, t).z;
      mine = (z & 0xffff) <= seg && seg <= (z >> 16);
    }
    return __ballot_sync(0xffffffffu, mine);
  };

  if (misaligned || idle) {
    // nothing was started
  } else if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(PR_REGS_LIGHT));
    if (warp == 0) {
      // ------------------------------------------------------------- TMA producer
      uint32_t n_loaded = 0;                                    // panels so far; stage = panel % 3
      bool ok = true;
      if (elect_one()) { tma_prefetch_desc(&map_blocks); tma_prefetch_desc(&map_uk); tma_prefetch_desc(&map_uv); }
      for (int i0 = blockIdx.x; i0 < n_items && ok; i0 += 32 * step) {
        for (unsigned m = lookup(i0); m && ok; m &= m - 1) {
          const int i = i0 + (__ffs(m) - 1) * step;
          int side, t;
          const int4 en = entry(i, side, t);
          const int cls = en.x & 0xff, n0 = (i % n_slabs) * NS;
          if (elect_one()) {
            const CUtensorMap* mu = side ? &map_uv : &map_uk;
            for (int p = 0; p < cls; ++p) {
              const uint32_t n = n_loaded + p, st = n % PR_STAGES, ph = (n / PR_STAGES) & 1u;
              if (!(ok = mbar_wait_thin(empty + 8 * st, ph ^ 1u, abort_flag))) break;
              mbar_expect_tx(full + 8 * st, PR_A_BYTES + (uint32_t)NS * 128u);
              const uint32_t dst = s0 + st * PR_STAGE_BYTES;
              tma_load_2d(dst, &map_blocks, full + 8 * st, 0, (en.y + p) * TILE);
              for (int at = 0; at < NS / 64; ++at) tma_load_2d(dst + PR_A_BYTES + at * PR_ATOM_BYTES, mu, full + 8 * st, n0 + at * 64, p * PANEL);
            }
          }
          __syncwarp();
          n_loaded += cls;
          ok = __all_sync(0xffffffffu, ok);
        }
      }
      if (!ok)                                                  // let copies in flight land before the CTA goes away
        for (uint32_t i = 0; i < PR_STAGES && i < n_loaded; ++i) {
          const uint32_t n = n_loaded - 1 - i;
          mbar_wait_drain(full + 8 * (n % PR_STAGES), (n / PR_STAGES) & 1u);
        }
    } else if (warp == 1) {
      // ------------------------------------------------------------- MMA issuer
      const uint32_t idesc = idesc_f16(BF16 ? 1 : 0, 128, NS) | (1u << 16);           // B MN-major
      uint32_t n_used = 0, ac = 0;
      bool ok = true;
      for (int i0 = blockIdx.x; i0 < n_items && ok; i0 += 32 * step) {
        for (unsigned m = lookup(i0); m && ok; m &= m - 1) {
          const int i = i0 + (__ffs(m) - 1) * step;
          int side, t;
          const int cls = entry(i, side, t).x & 0xff, len = pr_chain(side);
          if (elect_one()) {
            for (int p = 0; p < cls && ok; ++p) {
              const uint32_t chain = ac + p / len, buf = chain & 1u;
              if (p % len == 0) {
                if (!(ok = mbar_wait(acc_empty + 8 * buf, ((chain >> 1) & 1u) ^ 1u, abort_flag))) break;
                fence_after_sync();
              }
              const uint32_t n = n_used + p, st = n % PR_STAGES, ph = (n / PR_STAGES) & 1u;
              if (!(ok = mbar_wait_thin(full + 8 * st, ph, abort_flag))) break;
              fence_after_sync();
              const uint32_t sa = s0 + st * PR_STAGE_BYTES, sb = sa + PR_A_BYTES;
#pragma unroll
              for (int ks = 0; ks < 4; ++ks) {
                const uint32_t a_lo = kmajor_sw128_desc_lo(sa) + 2 * ks;
                const uint32_t b_lo = (((sb + ks * 2048u) >> 4) & 0x3fffu) | ((PR_ATOM_BYTES >> 4) << 16);
                mma_f16_ss(tmem_base + buf * 256, ((uint64_t)KMAJOR_SW128_DESC_HI << 32) | a_lo, ((uint64_t)KMAJOR_SW128_DESC_HI << 32) | b_lo,
                           idesc, (p % len > 0 || ks > 0) ? 1u : 0u);
              }
              mma_commit(empty + 8 * st);
              if (p % len == len - 1 || p == cls - 1) mma_commit(acc_full + 8 * buf);
            }
          }
          __syncwarp();
          n_used += cls;
          ac += (cls + len - 1) / len;
          ok = __all_sync(0xffffffffu, ok);
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(PR_REGS_EPI));
    // ------------------------------------------------------------- epilogue
    const int ew = warp - 4, quarter = warp & 3, hf = ew >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    unsigned char* stage = out_stage + ew * PR_OUT_BYTES;       // [high | low][32 rows][128 bytes]
    const size_t plane = (size_t)a.seg_rows * 256;              // bytes of one part of one head
    const int heads = NS / 128;
    const int* kpos = v.aux(layer, 0);
    const int seg0 = seg * a.seg_rows;
    // rows behind a sequence's last one, up to the next multiple of 128: their weights are zero, so their values must be finite
    for (int u = blockIdx.x; u < a.n_u; u += step) {
      const int r0 = a.base[u] + a.rows[u], r1 = a.base[u] + (a.rows[u] + TILE - 1) / TILE * TILE;
      if (r0 == r1 || r0 < seg0 || r0 >= seg0 + a.seg_rows) continue;
      for (int i = tid - 128; i < (r1 - r0) * 32 * v.Hkv; i += 256) {
        const int g = i / ((r1 - r0) * 32), rem = i - g * (r1 - r0) * 32, part = 2 + rem / ((r1 - r0) * 16), w = rem % ((r1 - r0) * 16);
        *reinterpret_cast<uint4*>(a.seg_buf + (g * 4 + part) * plane + (size_t)(r0 - seg0) * 256 + (size_t)w * 16) = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    uint32_t ac = 0;
    bool ok = true;
    const float vscale = a.vscale[0];
    // what an item's rows need from the tables; fetched an item ahead, so that the reads do not add up at its start
    int side = 0, t = 0, cls = 0, place = -1, pos = 0;
    auto fetch = [&](int i) {
      cls = entry(i, side, t).x & 0xff;
      place = (side ? a.vrow : a.krow_out)[(size_t)t * TILE + row];                      // rows past the tile's last token hold -1
      pos = side ? 0 : kpos[(size_t)t * TILE + row];
    };
    for (int i0 = blockIdx.x; i0 < n_items && ok; i0 += 32 * step) {
      unsigned m = lookup(i0);
      if (m) fetch(i0 + (__ffs(m) - 1) * step);
      for (; m; m &= m - 1) {
        const int i = i0 + (__ffs(m) - 1) * step;
        const int now_side = side, now_t = t, chains = (cls + pr_chain(side) - 1) / pr_chain(side), now_pos = pos;
        const int g0 = (i % n_slabs) * heads;
        int local = place - seg0;
        if (place < 0 || local < 0 || local >= a.seg_rows) local = -1;
        if (const unsigned rest = m & (m - 1)) fetch(i0 + (__ffs(rest) - 1) * step);
        auto stage_piece = [&](int piece, const uint32_t* hi, const uint32_t* lo) {      // 16 bytes of this thread's row, both parts
          unsigned char* d = stage + lane * 128 + ((piece ^ (lane & 7)) << 4);
          *reinterpret_cast<uint4*>(d) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          *reinterpret_cast<uint4*>(d + 4096) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        };
        // The warp's 32 half rows: four whole 128-byte pieces per instruction.  All of a part's reads go out before its first store:
        // with two warps per scheduler one read after the other cost the epilogue more than its arithmetic.
        auto rows_out = [&](int g, int half) {
          __syncwarp();
          unsigned char* dst = a.seg_buf + (g * 4 + now_side * 2) * plane + half * 128 + (lane & 7) * 16;
          int lr[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) lr[k] = __shfl_sync(0xffffffffu, local, 4 * k + (lane >> 3));
#pragma unroll
          for (int part = 0; part < 2; ++part) {
            uint4 w[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const int r = 4 * k + (lane >> 3);
              w[k] = *reinterpret_cast<const uint4*>(stage + part * 4096 + r * 128 + (((lane & 7) ^ (r & 7)) << 4));
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
              if (lr[k] >= 0) *reinterpret_cast<uint4*>(dst + part * plane + (size_t)lr[k] * 256) = w[k];
          }
          __syncwarp();
        };
        auto wait_chain = [&](uint32_t n) -> bool {
          const bool got = __all_sync(0xffffffffu, mbar_wait(acc_full + 8 * (n & 1u), (n >> 1) & 1u, abort_flag));
          fence_after_sync();
          return got;
        };
        auto free_chain = [&](uint32_t n) {
          fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_empty + 8 * (n & 1u));
        };
        if (!now_side) {
          // K: this thread's half of the RoPE frequencies; dims 32 hf + 8 c .. + 7 and the eight 64 above them at a time.
          // cos / sin of (position, frequency pair) by the angle-addition formulas from the two table rows.
          const float4* __restrict__ th = v.rope_hi + (size_t)((now_pos >> 4) & (ROPE_HI - 1)) * 32 + hf * 16;
          const float4* tl = sRope + (now_pos & 15) * PR_ROPE_STRIDE + hf * 16;
          uint64_t cs[16], sn[16];
          {
            float4 h4[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) h4[k] = __ldg(th + k);
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const float4 l4 = tl[k];
              const uint64_t ch = pk2(h4[k].x, h4[k].y), sh = pk2(h4[k].z, h4[k].w), cl = pk2(l4.x, l4.y), sl = pk2(l4.z, l4.w);
              cs[k] = sub2(mul2(ch, cl), mul2(sh, sl));
              sn[k] = fma2(sh, cl, mul2(ch, sl));
            }
          }
          ok = wait_chain(ac);
          if (ok && chains == 2) ok = wait_chain(ac + 1);
          if (!ok) break;
          for (int hh = 0; hh < heads; ++hh) {
            const uint32_t src = lane_addr + (ac & 1u) * 256 + hh * 128 + hf * 32, src2 = lane_addr + ((ac + 1) & 1u) * 256 + hh * 128 + hf * 32;
            uint32_t va[16], vb[16];                             // eight dims and the eight 64 above them; the next ones on their way
            tmem_ld8(src, va);
            tmem_ld8(src + 64, va + 8);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              uint32_t* x = (c & 1) ? vb : va;
              uint32_t* nx = (c & 1) ? va : vb;
              if (chains == 2) {
                uint32_t y[16];
                tmem_ld8(src2 + 8 * c, y);
                tmem_ld8(src2 + 64 + 8 * c, y + 8);
                tmem_ld_wait();
#pragma unroll
                for (int k = 0; k < 16; ++k) x[k] = __float_as_uint(__uint_as_float(x[k]) + __uint_as_float(y[k]));
              } else {
                tmem_ld_wait();
              }
              if (c < 3) {
                tmem_ld8(src + 8 * (c + 1), nx);
                tmem_ld8(src + 64 + 8 * (c + 1), nx + 8);
              } else if (hh == heads - 1) {
                free_chain(ac);
                if (chains == 2) free_chain(ac + 1);
              }
              uint32_t hi[8], lo[8];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const uint64_t L = pk2u(x[2 * k], x[2 * k + 1]), H = pk2u(x[8 + 2 * k], x[9 + 2 * k]);
                const uint64_t rl = sub2(mul2(L, cs[4 * c + k]), mul2(H, sn[4 * c + k])), rh = fma2(L, sn[4 * c + k], mul2(H, cs[4 * c + k]));
                split_pair_16<false>(rl, hi[k], lo[k]);
                split_pair_16<false>(rh, hi[4 + k], lo[4 + k]);
              }
              if (v.debug) {                                     // TWKV_DEBUG: a rotated key beyond the f16 range was clamped
                bool sat = false;
#pragma unroll
                for (int k = 0; k < 8; ++k) sat |= (hi[k] & 0x7fffu) == 0x7bffu || ((hi[k] >> 16) & 0x7fffu) == 0x7bffu;
                if (sat && local >= 0) set_status(v, TWKV_ERR_DEVICE_CHECK);
              }
              // keys are stored in the order in which decode attention contracts them (pairs of pieces 64 dims apart), so that the
              // sums round alike
              stage_piece(2 * c, hi, lo);
              stage_piece(2 * c + 1, hi + 4, lo + 4);
            }
            rows_out(g0 + hh, hf);
          }
          ac += chains;
        } else {
          // V, summed over the chains.  A thread takes its row of head hf whole, both halves, so that it sees the row's largest value by
          // itself (finding it at a barrier of two half rows cost 7 % of the kernel); with one head per slab the two sets of warps take
          // turns, tile by tile.
          uint32_t x[2][64];
          for (int ch = 0; ch < chains; ++ch, ++ac) {
            if (!(ok = wait_chain(ac))) break;
#pragma unroll
            for (int p = 0; p < 2; ++p) {
              const uint32_t src = lane_addr + (ac & 1u) * 256 + (heads == 2 ? hf * 128 : 0) + p * 64;
              if (ch == 0) {
                tmem_ld32(src, x[p]);
                tmem_ld32(src + 32, x[p] + 32);
              } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  uint32_t y[16];
                  tmem_ld16(src + 16 * e, y);
                  tmem_ld_wait();
#pragma unroll
                  for (int k = 0; k < 16; ++k) x[p][16 * e + k] = __float_as_uint(__uint_as_float(x[p][16 * e + k]) + __uint_as_float(y[k]));
                }
              }
            }
            tmem_ld_wait();
            free_chain(ac);
          }
          if (!ok) break;
          float mx[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int k = 0; k < 128; k += 2) mx[(k >> 1) & 3] = max_abs3(mx[(k >> 1) & 3], x[k >> 6][k & 63], x[k >> 6][(k & 63) + 1]);
          const float top = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * vscale;
          int e = 0;                                             // (an infinite row is left as it is)
          if ((top > PR_V_MAX && top < INFINITY) || (top < PR_V_MIN && top > 0.f))
            e = max((int)(__float_as_uint(top) >> 23) - 127 + (top < 1.f ? 3 : -14), PR_EXP_MIN);
          const int g = heads == 2 ? g0 + hf : g0;
          if (heads == 1 && (now_t & 1) != hf) local = -1;           // (leaving the branch here instead cost 12 % of the kernel in spills)
          if (local >= 0) {
            a.vexp[(size_t)g * a.seg_rows + local] = (signed char)e;
            if (e != 0) a.vflag[(local / TILE) * v.Hkv + g] = seg + 1;
          }
          if (__any_sync(0xffffffffu, e != 0 || vscale != 1.f)) {
            const float f = __uint_as_float((uint32_t)(127 - e) << 23) * vscale;
#pragma unroll
            for (int k = 0; k < 128; ++k) x[k >> 6][k & 63] = __float_as_uint(__uint_as_float(x[k >> 6][k & 63]) * f);
          }
#pragma unroll
          for (int p = 0; p < 2; ++p) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              uint32_t hi[8], lo[8];
#pragma unroll
              for (int k = 0; k < 8; ++k) split_pair_16<false, false>(pk2u(x[p][16 * c + 2 * k], x[p][16 * c + 2 * k + 1]), hi[k], lo[k]);
              stage_piece(2 * c, hi, lo);
              stage_piece(2 * c + 1, hi + 4, lo + 4);
            }
            rows_out(g, p);
          }
        }
      }
    }
    tmem_ld_wait();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  if (warp == 1) tmem_dealloc(tmem_base, 512);
  if (tid == 0 && *abort_flag) set_status(v, misaligned ? TWKV_ERR_DEVICE_CHECK : TWKV_ERR_TIMEOUT);
}

// ------------------------------------------------------------------------------------------ attention
// One work item = (block of queries, KV head, split of the segment's rows).  A block is two tiles of 128 rows, row =
// (query, head of the group); their queries stay in shared memory, their accumulators in TMEM:
//   columns   0 .. 127 scores / weights of tile 0 | 128 .. 255 of tile 1 | 256 .. 383 output of tile 0 | 384 .. 511 of tile 1
// The weights overwrite the scores they come from (of every 16 columns the first 8 become high parts, the others low parts),
// and are the A operand of the second product from there.  Order of the products per key block j: O0 += P0 V(j), S0 = Q0
// K(j+1)^T, O1 += P1 V(j), S1 = Q1 K(j+1)^T, so that one tile's softmax runs beside the other's products; products of one
// thread retire in order, so S0 may overwrite P0 without a wait.
// The running maximum a row is scaled by moves only when it would grow by more than 2^8 (f16 holds 2^15), as FlashAttention-4
// describes it: the accumulator in TMEM is rescaled rarely, and by the softmax warps themselves.
// What bounds it: a tile's softmax plus its own products must fit beside the other tile's products (2 x 2560 tensor cycles per
// key block); eight warps per tile, thread = half a row.
// Warp roles (640 threads): 0 TMA producer, 1 MMA issuer, 4-11 softmax of tile 0, 12-19 softmax of tile 1.
constexpr int PA_THREADS = 640;
constexpr int PA_REGS_LIGHT = 64, PA_REGS_SOFTMAX = 104;        // 640 threads of 96 registers, divided again by warpgroup
constexpr int PA_STAGES = 5;                                    // 32-KiB stages: one part (high or low) of 128 keys or values
constexpr uint32_t PA_STAGE_BYTES = 32768, PA_PANEL_BYTES = 16384;
constexpr uint32_t PA_Q_BYTES = 2 * 32768;
constexpr uint32_t PA_X_BYTES = 2 * 2 * TILE * 4;               // [tile][half][row]: row maxima of a half; row sums at the end
constexpr uint32_t PA_SMEM = PA_Q_BYTES + PA_STAGES * PA_STAGE_BYTES + PA_X_BYTES + 8 * (2 * PA_STAGES + 8) + 16;
static_assert(PA_SMEM > CHAIN_TMEM_SMEM, "no other CTA with tensor memory beside this one");

__device__ __forceinline__ float ex2(float x) { float r; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x)); return r; }

struct PfItem { int first, cnt, tiles, g, split, blk, row_lo, key0, n_blk, dup; };

__device__ __forceinline__ PfItem pf_item(const DevView& v, const PfCall& a, int i, int seg) {
  PfItem it;
  const int per = v.Hkv * a.n_splits;
  it.blk = a.blk0 + a.blk_n - 1 - i / per;                      // late queries (they see most) first
  it.g = (i / a.n_splits) % v.Hkv;
  it.split = i % a.n_splits;
  const int2 q = a.blocks[it.blk];
  const int4 b = a.binfo[it.blk];
  it.first = q.x;
  it.cnt = q.y & 0x1ff;
  it.tiles = it.cnt * v.rep > TILE ? 2 : 1;
  it.dup = b.z;
  const int s0 = seg * a.seg_rows;
  const int lo = max(b.x, s0), hi = min(b.x + b.y, s0 + a.seg_rows);
  const int nb = hi > lo ? (hi - lo + TILE - 1) / TILE : 0;
  const int j0 = nb * it.split / a.n_splits, j1 = nb * (it.split + 1) / a.n_splits;
  it.row_lo = lo - s0 + j0 * TILE;                              // first row inside the segment buffer
  it.key0 = lo - b.x + j0 * TILE;                               // the same row, counted from the sequence's first
  it.n_blk = j1 - j0;
  return it;
}

// Sixteen consecutive outputs (element offset o) in the output type.
__device__ __forceinline__ void pf_store16(void* out, int out_dtype, size_t o, const float* x) {
  if (out_dtype == TWKV_F32) {
    float4* d = reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + o);
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] = make_float4(x[4 * k], x[4 * k + 1], x[4 * k + 2], x[4 * k + 3]);
  } else {
    unsigned w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (out_dtype == TWKV_BF16) asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[k]) : "f"(x[2 * k + 1]), "f"(x[2 * k]));
      else asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(w[k]) : "f"(x[2 * k + 1]), "f"(x[2 * k]));
    }
    uint4* d = reinterpret_cast<uint4*>(reinterpret_cast<unsigned short*>(out) + o);
    d[0] = make_uint4(w[0], w[1], w[2], w[3]);
    d[1] = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

template <bool BF16>
__global__ void __launch_bounds__(PA_THREADS, 1)
pf_attn_kernel(const __grid_constant__ CUtensorMap map_seg, DevView v, PfCall a, int seg, const unsigned short* q, void* out) {
  chain_start();
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t s0 = smem_addr(smem_raw);
  const bool misaligned = (s0 & 1023u) != 0;
  const uint32_t sQ = s0, sR = s0 + PA_Q_BYTES;
  float* sX = reinterpret_cast<float*>(smem_raw + PA_Q_BYTES + PA_STAGES * PA_STAGE_BYTES);
  unsigned char* tail = smem_raw + PA_Q_BYTES + PA_STAGES * PA_STAGE_BYTES + PA_X_BYTES;
  const uint32_t bars = smem_addr(tail);
  const uint32_t full = bars, empty = full + 8 * PA_STAGES, q_full = empty + 8 * PA_STAGES, s_full = q_full + 16, p_full = s_full + 16, o_done = p_full + 16;
  uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(tail + 8 * (2 * PA_STAGES + 8));
  volatile int* abort_flag = reinterpret_cast<int*>(s_tmem_base + 1);
  if (tid == 0) {
    for (int i = 0; i < PA_STAGES; ++i) { mbar_init(full + 8 * i, 1); mbar_init(empty + 8 * i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(q_full + 8 * i, 8); mbar_init(s_full + 8 * i, 1); mbar_init(p_full + 8 * i, 8); mbar_init(o_done + 8 * i, 1); }
    *abort_flag = misaligned ? 1 : 0;
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc(smem_addr(s_tmem_base), 512);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem_base = *s_tmem_base;
  const int n_items = a.blk_n * v.Hkv * a.n_splits;
  chain_wait();
  const bool whole = pf_whole(a), idle = pf_idle(a, seg);

  if (misaligned || idle) {
    // nothing was started
  } else if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(PA_REGS_LIGHT));
    if (warp == 0) {
      // ------------------------------------------------------------- TMA producer: K low, K high, V high, V low of every key block
      if (elect_one()) {
        tma_prefetch_desc(&map_seg);
        uint32_t st = 0, ph = 0, n_loaded = 0;
        bool ok = true;
        for (int i = blockIdx.x; i < n_items && ok; i += gridDim.x) {
          const PfItem it = pf_item(v, a, i, seg);
          for (int j = 0; j < it.n_blk && ok; ++j)
            for (int part = 0; part < 4; ++part) {
              if (!(ok = mbar_wait_thin(empty + 8 * st, ph ^ 1u, abort_flag))) break;
              mbar_expect_tx(full + 8 * st, PA_STAGE_BYTES);
              const int y = (it.g * 4 + (part < 2 ? part ^ 1 : part)) * a.seg_rows + it.row_lo + j * TILE;
              tma_load_2d(sR + st * PA_STAGE_BYTES, &map_seg, full + 8 * st, 0, y);
              tma_load_2d(sR + st * PA_STAGE_BYTES + PA_PANEL_BYTES, &map_seg, full + 8 * st, 64, y);
              ++n_loaded;
              if (++st == PA_STAGES) { st = 0; ph ^= 1u; }
            }
        }
        if (!ok)                                                // let copies in flight land before the CTA goes away
          for (uint32_t i = 0; i < PA_STAGES && i < n_loaded; ++i) {
            const uint32_t n = n_loaded - 1 - i;
            mbar_wait_drain(full + 8 * (n % PA_STAGES), (n / PA_STAGES) & 1u);
          }
      }
      __syncwarp();
    } else if (warp == 1) {
      // ------------------------------------------------------------- MMA issuer (one elected lane)
      if (elect_one()) {
        constexpr uint32_t idesc_s = idesc_f16(0, 128, 128);                            // f16 queries and keys, both K-major
        constexpr uint32_t idesc_o = idesc_f16(0, 128, 128) | (1u << 16);               // values MN-major
        uint32_t st = 0, ph = 0, qph[2] = {0, 0}, pph[2] = {0, 0};
        bool ok = true;
        // two consecutive stages (both parts of a block of keys or values)
        auto take = [&](uint32_t (&pair)[2]) -> bool {
          for (int k = 0; k < 2; ++k) {
            if (!mbar_wait_thin(full + 8 * st, ph, abort_flag)) return false;
            pair[k] = st;
            if (++st == PA_STAGES) { st = 0; ph ^= 1u; }
          }
          fence_after_sync();
          return true;
        };
        auto scores = [&](int h, const uint32_t (&k)[2]) {
          const uint32_t qa = kmajor_sw128_desc_lo(sQ + h * 32768u), d = tmem_base + h * 128;
#pragma unroll
          for (int part = 0; part < 2; ++part)                  // the low parts first: the sum is cut after every instruction
#pragma unroll
            for (int pn = 0; pn < 2; ++pn)
              mma_f16_ss_panel(d, qa + pn * (PA_PANEL_BYTES >> 4), kmajor_sw128_desc_lo(sR + k[part] * PA_STAGE_BYTES + pn * PA_PANEL_BYTES), idesc_s,
                               part + pn > 0 ? 1u : 0u);
          mma_commit(s_full + 8 * h);
        };
        auto values = [&](int h, const uint32_t (&vv)[2], bool first) {
          const uint32_t p = tmem_base + h * 128, d = tmem_base + 256 + h * 128;
#pragma unroll
          for (int c = 0; c < 3; ++c) {                         // high . low, low . high, high . high: the small ones first, as for the scores
            const uint32_t pa = p + (c == 1 ? 8 : 0);
            const uint32_t vb = (((sR + vv[c == 0] * PA_STAGE_BYTES) >> 4) & 0x3fffu) | ((PA_PANEL_BYTES >> 4) << 16);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
              mma_f16_ts(d, pa + 16 * ks, ((uint64_t)KMAJOR_SW128_DESC_HI << 32) | (vb + ks * 128u), idesc_o,
                         (c > 0 || ks > 0) ? 1u : (first ? 0u : 1u));
          }
          mma_commit(o_done + 8 * h);
        };
        for (int i = blockIdx.x; i < n_items && ok; i += gridDim.x) {
          const PfItem it = pf_item(v, a, i, seg);
          if (it.n_blk == 0) continue;                           // no hand-over of queries either, as in the softmax warps
          for (int h = 0; h < it.tiles && ok; ++h) { ok = mbar_wait(q_full + 8 * h, qph[h], abort_flag); qph[h] ^= 1u; }
          if (!ok) break;
          fence_after_sync();
          uint32_t kk[2], vv[2];
          if (!(ok = take(kk))) break;
          for (int h = 0; h < it.tiles; ++h) scores(h, kk);
          mma_commit(empty + 8 * kk[0]); mma_commit(empty + 8 * kk[1]);
          for (int j = 0; j < it.n_blk && ok; ++j) {
            if (!(ok = take(vv))) break;
            const bool more = j + 1 < it.n_blk;
            for (int h = 0; h < it.tiles; ++h) {
              if (!(ok = mbar_wait_thin(p_full + 8 * h, pph[h], abort_flag))) break;
              pph[h] ^= 1u;
              fence_after_sync();
              values(h, vv, j == 0);
              if (h == it.tiles - 1) { mma_commit(empty + 8 * vv[0]); mma_commit(empty + 8 * vv[1]); }
              if (more) {
                if (h == 0 && !(ok = take(kk))) break;
                scores(h, kk);
                if (h == it.tiles - 1) { mma_commit(empty + 8 * kk[0]); mma_commit(empty + 8 * kk[1]); }
              }
            }
          }
        }
      }
      __syncwarp();
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(PA_REGS_SOFTMAX));
    // ------------------------------------------------------------- softmax
    const int grp = (warp - 4) >> 2, h = grp >> 1, hf = grp & 1, quarter = warp & 3, row = quarter * 32 + lane;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const uint32_t tS = lane_addr + h * 128 + hf * 64, tO = lane_addr + 256 + h * 128 + hf * 64;
    unsigned char* sq = smem_raw + h * 32768 + hf * PA_PANEL_BYTES;
    const int pair_bar = 1 + h * 4 + quarter;                    // the two warps that share 32 rows
    float* xs = sX + h * 2 * TILE + row;
    const int rep = v.rep, QT = TILE / rep;
    // scores in powers of two; a negative scale goes into the queries, a zero one zeroes them (-inf masks need a positive factor)
    const float scale = v.sm_scale == 0.f ? 1.f : fabsf(v.sm_scale) * 1.44269504088896340736f;
    const unsigned flip = v.sm_scale < 0.f ? 0x80008000u : 0u, keep_q = v.sm_scale == 0.f ? 0u : 0xffffffffu;
    uint32_t sph = 0, oph = 0;                                   // phases of s_full and of the next o_done
    bool ok = true;
    for (int i = blockIdx.x; i < n_items && ok; i += gridDim.x) {
      const PfItem it = pf_item(v, a, i, seg);
      if (h >= it.tiles) continue;
      // An item without key blocks hands nothing over: nothing would hold these warps back, and two items ahead of the other tile
      // they would complete a phase of q_full that the issuer (which waits for the tiles in turn) has not seen.  With keys, o_done
      // keeps them within one item.
      if (it.n_blk > 0) {
        // this warp's half of its 32 query rows as the K-major operand, four rows per instruction
#pragma unroll 4
        for (int k = 0; k < 8; ++k) {
          const int r = quarter * 32 + 4 * k + (lane >> 3), k8 = lane & 7;
          const int ch = hf * 4 + (k8 >> 1) + 8 * (k8 & 1);        // the keys' order: pairs of pieces 64 dims apart
          const int ql = h * QT + r / rep;
          uint4 val = make_uint4(0u, 0u, 0u, 0u);
          if (ql < it.cnt)
            val = reinterpret_cast<const uint4*>(q + ((size_t)a.qrow[it.first + ql] * v.Hq + it.g * rep + r % rep) * HEAD_DIM)[ch];
          if constexpr (BF16) {
            const unsigned w[4] = {val.x, val.y, val.z, val.w};
            unsigned o[4];
            bool over = false;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xffff0000u);
              over |= !(fabsf(lo) <= 65504.f) || !(fabsf(hi) <= 65504.f);
              o[e] = pack_f16x2_sat(lo, hi);
            }
            if (over) set_status(v, TWKV_ERR_DEVICE_CHECK);        // a bf16 query beyond the f16 range would be clamped
            val = make_uint4(o[0], o[1], o[2], o[3]);
          }
          val.x = (val.x ^ flip) & keep_q; val.y = (val.y ^ flip) & keep_q; val.z = (val.z ^ flip) & keep_q; val.w = (val.w ^ flip) & keep_q;
          *reinterpret_cast<uint4*>(sq + r * 128 + ((k8 ^ (r & 7)) << 4)) = val;
        }
        fence_proxy_async_smem();
        fence_before_sync();                                       // the previous item's accumulator has been read as well
        __syncwarp();
        if (lane == 0) mbar_arrive(q_full + 8 * h);
      }

      const int ql = h * QT + row / rep;
      const int vis = ql < it.cnt ? a.qvis[it.first + ql] : 0;
      const int qpos = it.dup && ql < it.cnt ? a.qpos[it.first + ql] : -1;
      float m = -INFINITY;
      uint64_t l2 = 0;                                           // two partial sums of this half's weights
      for (int j = 0; j < it.n_blk; ++j) {
        const int flag = a.vflag[((it.row_lo >> 7) + j) * v.Hkv + it.g];         // (on its way while the scores are waited for)
        ok = __all_sync(0xffffffffu, mbar_wait(s_full + 8 * h, sph, abort_flag));
        sph ^= 1u;
        fence_after_sync();
        uint32_t x[64];
        tmem_ld32(tS, x);
        tmem_ld32(tS + 32, x + 32);
        tmem_ld_wait();
        const int left = vis - (it.key0 + j * TILE) - hf * 64;   // columns of this half that the row sees (repeated positions: that hold a token)
        if (it.dup || __any_sync(0xffffffffu, left < 64)) {
          unsigned see[2];                                       // one bit per column
#pragma unroll
          for (int e = 0; e < 2; ++e) see[e] = left >= 32 * (e + 1) ? 0xffffffffu : (left <= 32 * e ? 0u : (1u << (left - 32 * e)) - 1u);
          if (it.dup) {
            const int* rp = a.rowpos + (size_t)seg * a.seg_rows + it.row_lo + j * TILE + hf * 64;
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll 1
              for (int c = 0; c < 32; ++c)
                if (32 * e + c < left && rp[32 * e + c] > qpos) see[e] &= ~(1u << c);
          }
#pragma unroll
          for (int c = 0; c < 64; ++c) x[c] = (see[c >> 5] >> (c & 31)) & 1u ? x[c] : 0xff800000u;
        }
        // Scaled rows: a score takes its row's power of two along, so that maximum and weights are those of weight x value; the
        // sum of the weights leaves it out again.
        const bool scaled = flag == seg + 1;
        auto exps = [&](int c) -> int4 {                          // of columns 16 c .. 16 c + 15
          return reinterpret_cast<const int4*>(a.vexp + (size_t)it.g * a.seg_rows + it.row_lo + j * TILE + hf * 64)[c];
        };
        if (scaled) {
          const float inv_scale = fminf(1.f / scale, 1e30f);
#pragma unroll
          for (int c = 0; c < 64; c += 16) {
            const int4 w = exps(c >> 4);
            const int e4[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int k = 0; k < 16; ++k) x[c + k] = __float_as_uint(__uint_as_float(x[c + k]) + (float)(signed char)(e4[k >> 2] >> (8 * (k & 3))) * inv_scale);
          }
        }
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int c = 0; c < 64; c += 8)
#pragma unroll
          for (int e = 0; e < 4; ++e) mx[e] = fmaxf(mx[e], fmaxf(__uint_as_float(x[c + e]), __uint_as_float(x[c + 4 + e])));
        float top = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
        // Both halves of a row scale by the same maximum.  The next scores arrive only when both warps have handed over these
        // weights, so a warp never overwrites a value that its partner still reads.  A wait that ran out in either warp ends
        // the loop in both: neither is left at a barrier.
        xs[hf * TILE] = top;
        if (!(ok = named_bar_and(pair_bar, 64, ok))) break;
        top = fmaxf(top, xs[(hf ^ 1) * TILE]) * scale;
        const bool grow = top > m + 8.f;                          // also the first finite maximum
        if (__any_sync(0xffffffffu, grow)) {
          const float m_new = grow ? top : m;
          const float f = m == m_new ? 1.f : ex2(m - m_new);      // 0 when there was no maximum yet
          m = m_new;
          l2 = mul2(l2, pk2(f, f));
          if (j > 0) {
            // the previous block's product (a wait that ran out has raised the abort flag and ends the loop at the next barrier)
            const bool got = __all_sync(0xffffffffu, mbar_wait(o_done + 8 * h, oph ^ 1u, abort_flag));
            fence_after_sync();
            if (got) {
#pragma unroll 1
              for (int c = 0; c < 8; ++c) {
                uint32_t o[8];
                tmem_ld8(tO + 8 * c, o);
                tmem_ld_wait();
#pragma unroll
                for (int k = 0; k < 8; ++k) o[k] = __float_as_uint(__uint_as_float(o[k]) * f);
                tmem_st8(tO + 8 * c, o);
              }
            }
          }
        }
        const float mu = m == -INFINITY ? 0.f : m;
        const uint64_t nm2 = pk2(-mu, -mu), sc2 = pk2(scale, scale);
        auto weights = [&](auto with_exps) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint32_t w[16];                                      // 8 columns of high parts, 8 of low ones, over the scores they come from
            int4 ex = make_int4(0, 0, 0, 0);
            if constexpr (with_exps.value) ex = exps(c);
            const int e4[4] = {ex.x, ex.y, ex.z, ex.w};
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              float p0, p1;
              unpk2(fma2(pk2u(x[16 * c + 2 * k], x[16 * c + 2 * k + 1]), sc2, nm2), p0, p1);
              const uint64_t p = pk2(ex2(p0), ex2(p1));
              if constexpr (with_exps.value) {
                float f[2];
#pragma unroll
                for (int b = 0; b < 2; ++b) {                     // (bytes of rows that hold no token may be anything: their weight is 0)
                  const int e = min(max((int)(signed char)(e4[k >> 1] >> (16 * (k & 1) + 8 * b)), PR_EXP_MIN), PR_EXP_MAX);
                  f[b] = __uint_as_float((uint32_t)(127 - e) << 23);
                }
                l2 = fma2(p, pk2(f[0], f[1]), l2);
              } else {
                l2 = add2(l2, p);
              }
              split_pair_16<false>(p, w[k], w[8 + k]);
            }
            tmem_st16(tS + 16 * c, w);
          }
        };
        if (scaled) weights(std::true_type{}); else weights(std::false_type{});
        tmem_st_wait();
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(p_full + 8 * h);
        oph ^= 1u;
      }
      float l = 0.f;
      if (it.n_blk > 0) {
        if (!ok) break;                                          // agreed by both warps above
        ok = __all_sync(0xffffffffu, mbar_wait(o_done + 8 * h, oph ^ 1u, abort_flag));
        fence_after_sync();
        float la, lb;
        unpk2(l2, la, lb);
        xs[hf * TILE] = la + lb;                                 // the row sum of both halves
        if (!(ok = named_bar_and(pair_bar, 64, ok))) break;
        l = xs[0] + xs[TILE];                                    // (read before this warp hands over the next item's queries)
      }
      if (whole) {
        // This is the whole result.  A thread writes its row's 64 columns itself (4096-token prompt in four
        // calls 783 -> 751 us, five short prompts 204 -> 189 against partial results and the combine kernel).
        const float inv = l == 0.f ? 0.f : a.vscale[1] / l;      // 0: no token seen; a NaN stays one
        const bool mine = ql < it.cnt;
        const size_t o0 = mine ? ((size_t)a.qrow[it.first + ql] * v.Hq + it.g * rep + row % rep) * HEAD_DIM + hf * 64 : 0;
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          float x[16];
#pragma unroll
          for (int k = 0; k < 16; ++k) x[k] = 0.f;
          if (it.n_blk > 0) {                                    // (the same for the whole warp, as the load demands)
            tmem_ld16(tO + 16 * c, reinterpret_cast<uint32_t*>(x));
            tmem_ld_wait();
#pragma unroll
            for (int k = 0; k < 16; ++k) x[k] *= inv;
          }
          if (mine) pf_store16(out, v.out_dtype, o0 + 16 * c, x);
        }
        continue;
      }
      // the item's partial result, joined with what earlier segments left; column-major, so that a warp's rows lie together
      float* part = a.slots + ((((size_t)(it.blk - a.blk0) * v.Hkv + it.g) * a.n_splits + it.split) * 2 + h) * (130 * TILE) + row;
      if (it.n_blk > 0) {
        float wo = 1.f, wp = 0.f;
        if (seg > 0) {
          const float mp = part[128 * TILE], lp = part[129 * TILE];
          named_bar_sync(pair_bar, 64);                          // both halves have read them
          if (lp != 0.f) {                                       // (also a NaN, which the result must show)
            const float mm = fmaxf(m, mp);
            wo = m == -INFINITY ? 0.f : ex2(m - mm);
            wp = ex2(mp - mm);
            l = l * wo + lp * wp;
            m = mm;
          }
        }
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          uint32_t o[16];
          tmem_ld16(tO + 16 * c, o);
          tmem_ld_wait();
          float* pc = part + (size_t)(hf * 64 + 16 * c) * TILE;
          if (wp > 0.f) {
#pragma unroll
            for (int k = 0; k < 16; ++k) pc[k * TILE] = __uint_as_float(o[k]) * wo + pc[k * TILE] * wp;
          } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) pc[k * TILE] = __uint_as_float(o[k]);
          }
        }
        if (hf == 0) { part[128 * TILE] = m; part[129 * TILE] = l; }
      } else if (seg == 0 && hf == 0) {
        part[128 * TILE] = -INFINITY; part[129 * TILE] = 0.f;
      }
    }
    tmem_ld_wait();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  if (warp == 1) tmem_dealloc(tmem_base, 512);
  if (tid == 0 && *abort_flag) set_status(v, misaligned ? TWKV_ERR_DEVICE_CHECK : TWKV_ERR_TIMEOUT);
}

// Joins the splits of one tile of rows and writes the queries' outputs.  One CTA per (block of queries, KV head, tile, 32
// columns); a thread owns one row of 16 of the columns, so reads are coalesced along the rows; rows leave through shared
// memory.
template <int OUT>
__global__ void __launch_bounds__(256) pf_combine_kernel(DevView v, PfCall a, void* out) {
  __shared__ float s[TILE][33];
  chain_start();
  chain_wait();
  if (pf_whole(a)) return;
  const int c0 = (blockIdx.x & 3) * 32, h = (blockIdx.x >> 2) & 1, bg = blockIdx.x >> 3, g = bg % v.Hkv, blk = bg / v.Hkv;
  const int2 q = a.blocks[a.blk0 + blk];
  const int cnt = q.y & 0x1ff, rep = v.rep, QT = TILE / rep;
  const int rows = min(TILE, (cnt - h * QT) * rep);
  if (rows <= 0) return;
  const int tid = threadIdx.x, row = tid & (TILE - 1), cc = (tid >> 7) * 16;
  const size_t stride = (size_t)2 * 130 * TILE;
  const float* part = a.slots + (((size_t)blk * v.Hkv + g) * a.n_splits * 2 + h) * (130 * TILE) + row;
  float m = -INFINITY, l = 0.f;
  float acc[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) acc[c] = 0.f;
  for (int k = 0; k < a.n_splits; ++k) {
    const float lk = part[k * stride + 129 * TILE], mk = part[k * stride + 128 * TILE];
    if (lk == 0.f) continue;                                      // nothing seen; a NaN goes into the sum
    float x[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) x[c] = part[k * stride + (c0 + cc + c) * TILE];
    const float mn = fmaxf(m, mk), wo = ex2(m - mn), wk = ex2(mk - mn);     // first split: wo = 0
    l = l * wo + lk * wk;
#pragma unroll
    for (int c = 0; c < 16; ++c) acc[c] = acc[c] * wo + x[c] * wk;
    m = mn;
  }
  const float inv = l == 0.f ? 0.f : a.vscale[1] / l;
#pragma unroll
  for (int c = 0; c < 16; ++c) s[row][cc + c] = acc[c] * inv;
  __syncthreads();
  for (int i = tid; i < rows * 4; i += 256) {                     // eight columns of one row
    const int r = i >> 2, c8 = (i & 3) * 8;
    const int ql = h * QT + r / rep;
    const size_t o = ((size_t)a.qrow[q.x + ql] * v.Hq + g * rep + r % rep) * HEAD_DIM + c0 + c8;
    const float* x = &s[r][c8];
    if constexpr (OUT == TWKV_F32) {
      float4* d = reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + o);
      d[0] = make_float4(x[0], x[1], x[2], x[3]);
      d[1] = make_float4(x[4], x[5], x[6], x[7]);
    } else {
      unsigned w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if constexpr (OUT == TWKV_BF16) asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[k]) : "f"(x[2 * k + 1]), "f"(x[2 * k]));
        else asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(w[k]) : "f"(x[2 * k + 1]), "f"(x[2 * k]));
      }
      *reinterpret_cast<uint4*>(reinterpret_cast<unsigned short*>(out) + o) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// ------------------------------------------------------------------------------------------ host side
cudaError_t launch_pf_tables(const DevView& v, const PfCall& a, int layer, int sm_count, cudaStream_t st) {
  ProfScope ps(TWKV_K_PLAN, st);
  const int zc = (a.n_words + 8191) / 8192, qctas = (a.n_blocks + 31) / 32;
  const int qc = qctas > sm_count ? sm_count : qctas;
  const dim3 b(1024), one(1);
  cudaError_t e = launch_chained(pf_init_kernel, dim3(zc < 1 ? 1 : (zc > sm_count ? sm_count : zc)), b, one, 0, st, v, a);
  if (e == cudaSuccess) e = launch_chained(pf_bits_kernel, dim3(sm_count), b, one, 0, st, v, a, layer);
  if (e == cudaSuccess) e = launch_chained(pf_scan_kernel, dim3(a.n_u), b, one, 0, st, v, a, layer);
  if (e == cudaSuccess) e = launch_chained(pf_rows_kernel, dim3(sm_count + qc + 1), b, one, 0, st, v, a, layer, qc);
  if (e != cudaSuccess) return e;
  count_launch(4);
  return cudaGetLastError();
}

template <bool BF16>
static cudaError_t launch_pf_segment_t(const DevView& v, const PfCall& a, const PfMaps& maps, int layer, int seg, const void* q, void* out, int sm_count, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(pf_recon_kernel<BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PR_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(pf_attn_kernel<BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PA_SMEM);
  if (e != cudaSuccess) return e;
  {
    ProfScope ps(TWKV_K_KSCORE, st);
    e = launch_chained(pf_recon_kernel<BF16>, dim3(sm_count), dim3(PR_THREADS), dim3(1), PR_SMEM, st, maps.blocks, maps.uk, maps.uv, v, a, layer, seg);
    if (e != cudaSuccess) return e;
  }
  const int n_items = a.blk_n * v.Hkv * a.n_splits;
  {
    ProfScope ps(TWKV_K_VACC, st);
    e = launch_chained(pf_attn_kernel<BF16>, dim3(n_items < sm_count ? n_items : sm_count), dim3(PA_THREADS), dim3(1), PA_SMEM, st, maps.seg, v, a, seg,
                       reinterpret_cast<const unsigned short*>(q), out);
    if (e != cudaSuccess) return e;
  }
  count_launch(2);
  return cudaGetLastError();
}
cudaError_t launch_pf_segment(const DevView& v, const PfCall& a, const PfMaps& maps, int layer, int seg, const void* q, void* out, int sm_count, cudaStream_t st) {
  return v.dtype == TWKV_BF16 ? launch_pf_segment_t<true>(v, a, maps, layer, seg, q, out, sm_count, st)
                              : launch_pf_segment_t<false>(v, a, maps, layer, seg, q, out, sm_count, st);
}

cudaError_t launch_pf_combine(const DevView& v, const PfCall& a, void* out, cudaStream_t st) {
  ProfScope ps(TWKV_K_MERGE, st);
  const int grid = a.blk_n * v.Hkv * 8;
  auto kernel = v.out_dtype == TWKV_F32 ? pf_combine_kernel<TWKV_F32> : v.out_dtype == TWKV_BF16 ? pf_combine_kernel<TWKV_BF16> : pf_combine_kernel<TWKV_F16>;
  const cudaError_t e = launch_chained(kernel, dim3(grid), dim3(256), dim3(1), 0, st, v, a, out);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace twkv

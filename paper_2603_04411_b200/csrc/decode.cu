// Decode attention over the mixed-rank cache (Eq. 3, reshape to heads, RoPE, softmax attention).
//
//   plan_kernel    sequence id -> query slot map, running-max reset, K-tile work list; cut points of every
//                  sequence's V tiles into the splits of the V pass; K slot -> V slot links of the sequences' tokens
//   kscore_tc_kernel (kscore_tc.cu)  per K tile: Kbar = X^_K U_K^-1, RoPE by stored position,
//                  s = q . Kbar * scale for the GQA group, scores to scratch, per-sequence max
//   vacc_tc_kernel (vacc_tc.cu)  per (sequence, split): p = exp(s - max), acc += p^T X^_V in spectral
//                  space (tcgen05), l = sum p
//   merge_kernel   sum of the splits, out_h = (acc_h / l_h) U_V^-1[:, head slice]
//
// V is never reconstructed per token: by linearity of Eq. 3 the weighted sum is taken in
// spectral space and projected once.
#include "twkv_dev.h"
#include "mma_util.cuh"
#include "tc_util.cuh"

namespace twkv {

// ------------------------------------------------------------------------------ plan
// One CTA: sequence id -> query slot map, running-max reset, and the K-score work list: the K tiles
// of the listed sequences in class order (widest first, inside a class in table order), compacted
// with block-wide scans so the order does not depend on thread timing.  For the CTA-pair kernel the list
// is rewritten as items of two tiles of one class.  The list is then cut into n_cta contiguous pieces of
// about equal estimated cost, so a CTA (pair) of the K-score kernel mostly stays inside one (class, sequence) run.
__device__ __forceinline__ unsigned ktile_cost(int cls) {
  // cycles per tile of the K-score kernel by rank class: a least-squares fit, one coefficient per class, of every CTA's busy
  // time to its tile counts on the benchmark's mix of classes (8 KV heads, CTA pairs; residual 1.3 us rms of 330): a fixed
  // part (rotation factors, the per-slab epilogue and score products) plus a per-panel part, an odd panel count costing a
  // little more than the even one above it saves; classes above 8 run as two passes.  Only the ratios matter.
  constexpr unsigned kCost[TWKV_MAX_CLASSES] = {14300u, 16600u, 18600u, 19500u, 22100u, 23000u, 25400u, 26200u,
                                                38800u, 38700u, 42000u, 42800u, 45600u, 45800u, 49300u, 50700u};
  return kCost[min(max(cls, 1), TWKV_MAX_CLASSES) - 1];
}

// Cut points of one sequence's V tile list into n_splits contiguous ranges of about equal cost (a tile costs its
// panels plus its score rows, counted in 512-byte units): the V pass is bound by the bytes a CTA reads, and tiles of
// classes 1 to 16 dealt out by count alone left the slowest CTA with half as much again as the mean.
// The list is taken in the stride order of vtile_stride(); cut[s] = number of tiles (in that order) whose inclusive cost
// prefix is <= s / n_splits of the total; split s takes positions cut[s] .. cut[s + 1] - 1 of that order.
__device__ void vsplit_plan(const DevView& v, int layer, const int* __restrict__ seq_ids, int qs, int n_splits) {
  __shared__ unsigned long long s_total, s_base;
  __shared__ unsigned s_ws[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int seq = seq_ids[qs];
  const int n = (seq >= 0 && seq < v.S) ? v.svc(layer)[seq] : 0;
  const int* list = v.svt(layer) + (size_t)(n > 0 ? seq : 0) * v.TPS;
  const int4* desc = v.desc(layer, 1);
  int* cut = v.vcut + (size_t)qs * (n_splits + 1);
  if (tid == 0) { s_total = 0ull; s_base = 0ull; }
  __syncthreads();
  unsigned mine = 0u;
  const long long stride = vtile_stride(n);
  for (int i = tid; i < n; i += blockDim.x) mine += 32u * (unsigned)desc[list[i]].y + (unsigned)v.Hq;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  if (lane == 0 && mine) atomicAdd(&s_total, (unsigned long long)mine);
  __syncthreads();
  const unsigned long long W = s_total, ns = (unsigned long long)n_splits;
  if (W == 0ull) {
    for (int s = tid; s <= n_splits; s += blockDim.x) cut[s] = 0;
    return;
  }
  for (int i0 = 0; i0 < n; i0 += blockDim.x) {
    const int i = i0 + tid;
    const unsigned w = i < n ? 32u * (unsigned)desc[list[(int)((i * stride) % n)]].y + (unsigned)v.Hq : 0u;
    unsigned inc = w;                                             // inclusive scan inside the warp, then over the warps
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned a = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += a;
    }
    if (lane == 31) s_ws[warp] = inc;
    __syncthreads();
    if (warp == 0) {
      unsigned wk = s_ws[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned a = __shfl_up_sync(0xffffffffu, wk, o);
        if (lane >= o) wk += a;
      }
      s_ws[lane] = wk;
    }
    __syncthreads();
    if (i < n) {
      const unsigned long long p = s_base + (warp ? s_ws[warp - 1] : 0u) + inc, e = p - w;
      // the splits whose boundary floor(s W / ns) falls in [e, p): they start at this tile
      for (unsigned long long s = (e * ns + W - 1ull) / W; s < ns && s * W / ns < p; ++s) cut[s] = i;
    }
    __syncthreads();
    if (tid == 0) s_base += s_ws[31];
    __syncthreads();
  }
  if (tid == 0) cut[n_splits] = n;
}

// K slot -> V slot of every token of one sequence (the V slots carry the opposite link): the K-score kernel stores a
// token's scores at its V slot, so that the V pass finds a tile's score rows next to each other.  CTA j of the vj CTAs of
// a sequence takes the V tiles j * 8 .. j * 8 + 7, then vj * 8 further on, eight tiles (1024 slots) at a time.
__device__ void vlink_plan(const DevView& v, int layer, const int* __restrict__ seq_ids, int qs, int j, int vj) {
  const int seq = seq_ids[qs];
  if (seq < 0 || seq >= v.S) return;
  const int n = v.svc(layer)[seq];
  const int* list = v.svt(layer) + (size_t)seq * v.TPS;
  const int4* desc = v.desc(layer, 1);
  const int* aux = v.aux(layer, 1);
  const int sub = threadIdx.x >> 7, slot = threadIdx.x & (TILE - 1);
  for (int t = j * 8 + sub; t < n; t += vj * 8) {
    const int vt = list[t];
    if (slot < desc[vt].z) v.kv_link[aux[(size_t)vt * TILE + slot]] = vt * TILE + slot;
  }
}

__global__ void __launch_bounds__(1024) plan_kernel(DevView v, int layer, const int* __restrict__ seq_ids, int n_seq, int n_cta, int pairs,
                                                    int n_splits, int vj) {
  if ((int)blockIdx.x > n_seq) {                                  // the last n_seq * vj CTAs: K slot -> V slot links
    const int idx = (int)blockIdx.x - 1 - n_seq;
    vlink_plan(v, layer, seq_ids, idx / vj, idx % vj, vj);
    return;
  }
  if (blockIdx.x > 0) {                                           // CTAs 1 .. n_seq: the V pass's split plan, one sequence each
    vsplit_plan(v, layer, seq_ids, (int)blockIdx.x - 1, n_splits);
    return;
  }
  __shared__ int s_cls_off[TWKV_MAX_CLASSES + 1], s_kcc[TWKV_MAX_CLASSES];
  __shared__ unsigned s_wsum[32];
  __shared__ unsigned s_base;                                     // entries kept so far
  __shared__ int s_keep[TWKV_MAX_CLASSES];                        // kept tiles per class run (run k = class NC - k)
  __shared__ int s_koff[TWKV_MAX_CLASSES + 1], s_ioff[TWKV_MAX_CLASSES + 1];    // start of run k in the tile list / in the item list
  __shared__ unsigned long long s_coff[TWKV_MAX_CLASSES + 1];     // estimated cost of everything before run k
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int s = tid; s < v.S; s += blockDim.x) v.qslot[s] = -1;
  if (tid < TWKV_MAX_CLASSES) s_keep[tid] = 0;
  // the class counts are read by sixteen threads at once (one thread reading them in a loop pays a memory round trip
  // per class)
  if (tid < v.NC) s_kcc[tid] = v.kcc(layer)[tid];
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int c = v.NC; c >= 1; --c) { s_cls_off[v.NC - c] = run; run += s_kcc[c - 1]; }    // widest class first
    s_cls_off[v.NC] = run;
    s_base = 0u;
  }
  __syncthreads();
  for (int i = tid; i < n_seq; i += blockDim.x) {
    const int s = seq_ids[i];
    if (s < 0 || s >= v.S) set_status(v, TWKV_ERR_INVALID_ARG);
    else v.qslot[s] = i;
  }
  for (int i = tid; i < n_seq * v.Hq; i += blockDim.x) v.seqmax[i] = 0u;
  __syncthreads();
  for (int i = tid; i < n_seq; i += blockDim.x) {
    const int s = seq_ids[i];
    if (s >= 0 && s < v.S && v.qslot[s] != i) set_status(v, TWKV_ERR_INVALID_ARG);   // duplicate id
  }
  const int4* desc = v.desc(layer, 0);
  const int* kct = v.kct(layer);
  const int n_all = s_cls_off[v.NC];
  constexpr int PL_BATCH = 4;                                     // list chunks of 1024 whose table reads are issued together
  for (int f0 = 0; f0 < n_all; f0 += 1024 * PL_BATCH) {
    // the three dependent reads (tile id -> descriptor -> query slot) of PL_BATCH chunks go out level by level
    int tile[PL_BATCH], run_[PL_BATCH];
    int4 d[PL_BATCH];
    int4 ent[PL_BATCH];
#pragma unroll
    for (int u = 0; u < PL_BATCH; ++u) {
      const int f = f0 + u * 1024 + tid;
      tile[u] = -1; run_[u] = 0;
      if (f < n_all) {
        int k = 0;
        while (f >= s_cls_off[k + 1]) ++k;
        run_[u] = k;
        tile[u] = kct[(size_t)(v.NC - k - 1) * v.NT + (f - s_cls_off[k])];
      }
    }
#pragma unroll
    for (int u = 0; u < PL_BATCH; ++u) d[u] = tile[u] >= 0 ? desc[tile[u]] : make_int4(0, 0, 0, 0);
#pragma unroll
    for (int u = 0; u < PL_BATCH; ++u)
      ent[u] = tile[u] >= 0 ? make_int4(tile[u], d[u].y | (d[u].z << 8), d[u].w, v.qslot[d[u].x]) : make_int4(0, 0, 0, -1);
#pragma unroll
    for (int u = 0; u < PL_BATCH; ++u) {
      if (f0 + u * 1024 >= n_all) break;                         // uniform across the CTA
      const int4 e = ent[u];
      const unsigned keep = e.w >= 0 ? 1u : 0u;
      unsigned ik = keep;                                         // inclusive scan inside the warp
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned a = __shfl_up_sync(0xffffffffu, ik, o);
        if (lane >= o) ik += a;
      }
      if (lane == 31) s_wsum[warp] = ik;
      __syncthreads();
      if (warp == 0) {
        unsigned wk = s_wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned a = __shfl_up_sync(0xffffffffu, wk, o);
          if (lane >= o) wk += a;
        }
        s_wsum[lane] = wk;                                        // inclusive over warps
      }
      __syncthreads();
      const unsigned pk = s_base + (warp ? s_wsum[warp - 1] : 0u) + ik - keep;      // exclusive position
      if (keep) { v.klist[pk] = e; atomicAdd(&s_keep[run_[u]], 1); }
      __syncthreads();
      if (tid == 0) s_base += s_wsum[31];
      __syncthreads();
    }
  }
  // class runs of the kept list: tiles, items (a pair item holds two tiles) and estimated cost before each run
  if (tid == 0) {
    int ko = 0, io = 0;
    unsigned long long co = 0ull;
    for (int k = 0; k < v.NC; ++k) {
      s_koff[k] = ko; s_ioff[k] = io; s_coff[k] = co;
      const int items = pairs ? (s_keep[k] + 1) / 2 : s_keep[k];
      ko += s_keep[k]; io += items;
      co += (unsigned long long)items * ktile_cost(v.NC - k);
    }
    s_koff[v.NC] = ko; s_ioff[v.NC] = io; s_coff[v.NC] = co;
    *v.klist_count = ko;
    v.cta_start[n_cta] = io;
  }
  __syncthreads();
  const int n_items = s_ioff[v.NC];
  const unsigned long long total = s_coff[v.NC];
  if (pairs) {
    for (int i = tid; i < n_items; i += blockDim.x) {
      int k = 0;
      while (i >= s_ioff[k + 1]) ++k;
      const int t0 = s_koff[k] + 2 * (i - s_ioff[k]);
      const int4 e0 = v.klist[t0];
      // a run of odd length ends with a filler: the same tile again, flagged so that its scores are dropped
      v.kpairs[2 * i] = e0;
      v.kpairs[2 * i + 1] = t0 + 1 < s_koff[k + 1] ? v.klist[t0 + 1] : make_int4(e0.x, e0.y | 0x80, e0.z, e0.w);
    }
  }
  // cut points: piece b starts at the item whose cost interval holds b / n_cta of the total (64-bit arithmetic; inside
  // a run every item costs the same, so the item follows from a division)
  for (int b = tid; b < n_cta; b += blockDim.x) {
    int start = 0;
    if (n_items > 0 && total > 0ull) {
      const unsigned long long key = (unsigned long long)b * total / (unsigned long long)n_cta;
      int k = 0;
      while (k + 1 < v.NC && s_coff[k + 1] <= key) ++k;
      const unsigned long long within = (key - s_coff[k]) / ktile_cost(v.NC - k);
      const int cap = s_ioff[k + 1] - s_ioff[k];
      start = s_ioff[k] + (int)(within < (unsigned long long)cap ? within : (unsigned long long)cap);
    }
    v.cta_start[b] = start;
  }
}

// -------------------------------------------------------------- merge + V projection
// A cluster of eight CTAs per (query slots, query heads of one KV head g): at most eight rows (slot, head).  CTA c takes
// the spectral components [c d/8, (c+1) d/8): it sums their splits, normalises, and multiplies by its rows of
// U_V^-1[:, g*128 .. g*128+127]; the eight partial [rows x 128] products meet through distributed shared memory, every CTA
// adding and writing 16 of the columns.  What bounds it is latency: one CTA doing a group's whole sum and product went
// through 256 KiB of U_V^-1 and every split by itself (29 us for one sequence of 1024 tokens with 64 splits, 23 us for 16
// sequences of 32768 tokens; now 6 and 9).  Empty splits are not read (the V pass does not write them).
constexpr int MG_THREADS = 256;
constexpr int MG_CL = 8;                             // CTAs of a cluster
constexpr int MG_ROWS = 8;

__device__ __forceinline__ float ld_cluster_f32(uint32_t addr) {
  float x;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(addr));
  return x;
}

template <bool BF16>
__global__ void __launch_bounds__(MG_THREADS)
merge_kernel(DevView v, const unsigned short* __restrict__ Uinv_v, int n_splits, int hp, int ns, int n_seq, void* __restrict__ out) {
  __shared__ float4 s_part[MG_THREADS];              // split sums per (split group, row, four components)
  __shared__ __align__(16) float s_acc[MG_ROWS * 128];    // [rows][d / 8] normalised
  __shared__ float s_red[4][MG_ROWS][128];
  __shared__ float s_out[MG_ROWS * 128];
  __shared__ float s_invl[MG_ROWS];
  // blockIdx.y = KV head g and which hp of its query heads; blockIdx.x / 8 = ns query slots that share the reads of U_V^-1
  const int c = tc::cluster_cta_rank();
  const int qs0 = (blockIdx.x / MG_CL) * ns, parts = v.rep / hp, g = blockIdx.y / parts, tid = threadIdx.x, lane = tid & 31;
  const int Hq = v.Hq, d_kv = v.d_kv;
  const int rows = min(ns, n_seq - qs0) * hp;
  const int head0 = g * v.rep + (blockIdx.y % parts) * hp;      // first query head of this CTA
  const int jn = d_kv / MG_CL, j0 = c * jn;                     // jn: a multiple of 16, at most 128
  // this thread's rows of U_V^-1 do not depend on the sums: their reads go out first (pair of columns dp, a quarter of the rows)
  const int dp = tid & 63, jg = tid >> 6, jr = jn / 4;
  const unsigned* ucol = reinterpret_cast<const unsigned*>(Uinv_v + (size_t)(j0 + jg * jr) * d_kv + g * HEAD_DIM) + dp;
  unsigned u[32];
#pragma unroll
  for (int t = 0; t < 32; ++t) u[t] = t < jr ? __ldg(ucol + (size_t)t * (d_kv / 2)) : 0u;
  // row sums over the splits: warp w takes row w, its lanes read the splits' parts together, lane 0 adds them in split order
  if ((tid >> 5) < rows) {
    const int r = tid >> 5, qs = qs0 + r / hp, head = head0 + r % hp;
    float l = 0.f;
    for (int s0 = 0; s0 < n_splits; s0 += 32) {
      const float mine = s0 + lane < n_splits ? v.part_l[((size_t)qs * n_splits + s0 + lane) * Hq + head] : 0.f;
      const int n = min(32, n_splits - s0);
      for (int s = 0; s < n; ++s) l += __shfl_sync(0xffffffffu, mine, s);
    }
    if (lane == 0) s_invl[r] = l > 0.f ? 1.f / l : 0.f;
  }
  // split sums: a thread owns four components of one row and every sg_n-th split, with eight reads in flight
  const int q4 = jn / 4, slots = rows * q4, sg_n = MG_THREADS / slots, sg = tid / slots, sl = tid - sg * slots;
  if (sg < sg_n) {
    const int r = sl / q4, qs = qs0 + r / hp;
    const float4* p = reinterpret_cast<const float4*>(v.part_acc + (((size_t)qs * n_splits) * Hq + head0 + r % hp) * d_kv + j0) + (sl - r * q4);
    const size_t stride = (size_t)Hq * d_kv / 4;
    const int* cut = v.vcut + (size_t)qs * (n_splits + 1);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = sg; s0 < n_splits; s0 += 8 * sg_n) {
      float4 t[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int s = s0 + k * sg_n;
        t[k] = s < n_splits && cut[s + 1] > cut[s] ? __ldg(p + (size_t)s * stride) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) { a.x += t[k].x; a.y += t[k].y; a.z += t[k].z; a.w += t[k].w; }
    }
    s_part[sg * slots + sl] = a;
  }
  __syncthreads();
  if (tid < slots) {
    float4 a = s_part[tid];
    for (int k = 1; k < sg_n; ++k) {                   // fixed order
      const float4 b = s_part[k * slots + tid];
      a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
    }
    const float il = s_invl[tid / q4];
    *reinterpret_cast<float4*>(s_acc + tid * 4) = make_float4(a.x * il, a.y * il, a.z * il, a.w * il);
  }
  __syncthreads();
  float o[MG_ROWS][2];
#pragma unroll
  for (int h = 0; h < MG_ROWS; ++h) { o[h][0] = 0.f; o[h][1] = 0.f; }
#pragma unroll
  for (int t = 0; t < 32; t += 4) {
    if (t >= jr) break;                                // jr is a multiple of 4
    float u0[4], u1[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) { u0[e] = to_f32<BF16>((unsigned short)(u[t + e] & 0xffffu)); u1[e] = to_f32<BF16>((unsigned short)(u[t + e] >> 16)); }
#pragma unroll
    for (int h = 0; h < MG_ROWS; ++h)
      if (h < rows) {
        const float4 a = *reinterpret_cast<const float4*>(s_acc + h * jn + jg * jr + t);
        o[h][0] += a.x * u0[0]; o[h][1] += a.x * u1[0];
        o[h][0] += a.y * u0[1]; o[h][1] += a.y * u1[1];
        o[h][0] += a.z * u0[2]; o[h][1] += a.z * u1[2];
        o[h][0] += a.w * u0[3]; o[h][1] += a.w * u1[3];
      }
  }
#pragma unroll
  for (int h = 0; h < MG_ROWS; ++h)
    if (h < rows) *reinterpret_cast<float2*>(&s_red[jg][h][2 * dp]) = make_float2(o[h][0], o[h][1]);
  __syncthreads();
  for (int i = tid; i < rows * 128; i += MG_THREADS)
    s_out[i] = ((s_red[0][i >> 7][i & 127] + s_red[1][i >> 7][i & 127]) + s_red[2][i >> 7][i & 127]) + s_red[3][i >> 7][i & 127];
  tc::cluster_sync_all();
  constexpr int CW = 128 / MG_CL;                      // columns this CTA writes
  if (tid < rows * CW) {
    const int h = tid / CW, dc = c * CW + tid % CW;
    const uint32_t at = tc::smem_addr(s_out + h * 128 + dc);
    float val = 0.f;
#pragma unroll
    for (int k = 0; k < MG_CL; ++k) val += ld_cluster_f32(tc::cluster_map(at, k));       // fixed order
    const int oslot = qs0 + h / hp;
    const size_t oi = ((size_t)(v.qmap ? v.qmap[oslot] : oslot) * Hq + head0 + h % hp) * HEAD_DIM + dc;
    if (v.out_dtype == TWKV_F32) reinterpret_cast<float*>(out)[oi] = val;
    else if (v.out_dtype == TWKV_BF16) reinterpret_cast<unsigned short*>(out)[oi] = from_f32<true>(val);
    else reinterpret_cast<unsigned short*>(out)[oi] = from_f32<false>(val);
  }
  tc::cluster_sync_all();                              // the partners have read this CTA's part
}

// The same for large batches: 32 rows per cluster share a CTA's slice of U_V^-1, staged in shared memory; thread = (pair of
// columns, a quarter of the rows).  With eight rows the reads of U_V^-1 (256 KiB per eight rows and KV head) bound it: 62 us
// for 64 sequences of 8192 tokens.
constexpr int MW_ROWS = 32;
constexpr int MW_SMEM = 128 * 128 * 2 + 2 * MW_ROWS * 128 * 4 + MW_ROWS * 4;

template <bool BF16>
__global__ void __launch_bounds__(MG_THREADS)
merge_wide_kernel(DevView v, const unsigned short* __restrict__ Uinv_v, int n_splits, int n_seq, void* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char mw_smem[];
  unsigned* s_u = reinterpret_cast<unsigned*>(mw_smem);                                // [d / 8][64] pairs of columns
  float* s_acc = reinterpret_cast<float*>(mw_smem + 128 * 128 * 2);                    // [rows][d / 8]
  float* s_out = s_acc + MW_ROWS * 128;                                                // [rows][128]
  float* s_invl = s_out + MW_ROWS * 128;
  const int c = tc::cluster_cta_rank(), g = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ns = MW_ROWS / v.rep, qs0 = (blockIdx.x / MG_CL) * ns;
  const int Hq = v.Hq, d_kv = v.d_kv, rep = v.rep;
  const int rows = min(ns, n_seq - qs0) * rep;
  const int jn = d_kv / MG_CL, j0 = c * jn;
  for (int i = tid; i < jn * 16; i += MG_THREADS) {                                    // 16-byte pieces of this CTA's rows of U_V^-1
    const uint4 w = __ldg(reinterpret_cast<const uint4*>(Uinv_v + (size_t)(j0 + (i >> 4)) * d_kv + g * HEAD_DIM) + (i & 15));
    reinterpret_cast<uint4*>(s_u)[i] = w;
  }
  for (int r = warp; r < rows; r += MG_THREADS / 32) {
    const int qs = qs0 + r / rep, head = g * rep + r % rep;
    float l = 0.f;
    for (int s0 = 0; s0 < n_splits; s0 += 32) {
      const float mine = s0 + lane < n_splits ? v.part_l[((size_t)qs * n_splits + s0 + lane) * Hq + head] : 0.f;
      const int n = min(32, n_splits - s0);
      for (int s = 0; s < n; ++s) l += __shfl_sync(0xffffffffu, mine, s);
    }
    if (lane == 0) s_invl[r] = l > 0.f ? 1.f / l : 0.f;
  }
  __syncthreads();
  const int q4 = jn / 4;
  for (int i = tid; i < rows * q4; i += MG_THREADS) {
    const int r = i / q4, qs = qs0 + r / rep;
    const float4* p = reinterpret_cast<const float4*>(v.part_acc + (((size_t)qs * n_splits) * Hq + g * rep + r % rep) * d_kv + j0) + (i - r * q4);
    const size_t stride = (size_t)Hq * d_kv / 4;
    const int* cut = v.vcut + (size_t)qs * (n_splits + 1);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < n_splits; s0 += 4) {
      float4 t[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        t[k] = s0 + k < n_splits && cut[s0 + k + 1] > cut[s0 + k] ? __ldg(p + (size_t)(s0 + k) * stride) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < 4; ++k) { a.x += t[k].x; a.y += t[k].y; a.z += t[k].z; a.w += t[k].w; }
    }
    const float il = s_invl[r];
    *reinterpret_cast<float4*>(s_acc + i * 4) = make_float4(a.x * il, a.y * il, a.z * il, a.w * il);
  }
  __syncthreads();
  const int dp = tid & 63, r0 = (tid >> 6) * (MW_ROWS / 4);
  if (r0 < rows) {
    float o[MW_ROWS / 4][2];
#pragma unroll
    for (int h = 0; h < MW_ROWS / 4; ++h) { o[h][0] = 0.f; o[h][1] = 0.f; }
    for (int t = 0; t < jn; t += 4) {
      float u0[4], u1[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const unsigned w = s_u[(t + e) * 64 + dp];
        u0[e] = to_f32<BF16>((unsigned short)(w & 0xffffu)); u1[e] = to_f32<BF16>((unsigned short)(w >> 16));
      }
#pragma unroll
      for (int h = 0; h < MW_ROWS / 4; ++h) {          // rows past the last hold whatever is in shared memory and are not written out
        const float4 a = *reinterpret_cast<const float4*>(s_acc + (r0 + h) * jn + t);
        o[h][0] += a.x * u0[0]; o[h][1] += a.x * u1[0];
        o[h][0] += a.y * u0[1]; o[h][1] += a.y * u1[1];
        o[h][0] += a.z * u0[2]; o[h][1] += a.z * u1[2];
        o[h][0] += a.w * u0[3]; o[h][1] += a.w * u1[3];
      }
    }
#pragma unroll
    for (int h = 0; h < MW_ROWS / 4; ++h) *reinterpret_cast<float2*>(s_out + (r0 + h) * 128 + 2 * dp) = make_float2(o[h][0], o[h][1]);
  }
  tc::cluster_sync_all();
  constexpr int CW = 128 / MG_CL;                      // columns this CTA writes
  for (int i = tid; i < rows * CW; i += MG_THREADS) {
    const int h = i / CW, dc = c * CW + i % CW;
    const uint32_t at = tc::smem_addr(s_out + h * 128 + dc);
    float val = 0.f;
#pragma unroll
    for (int k = 0; k < MG_CL; ++k) val += ld_cluster_f32(tc::cluster_map(at, k));       // fixed order
    const int oslot = qs0 + h / rep;
    const size_t oi = ((size_t)(v.qmap ? v.qmap[oslot] : oslot) * Hq + g * rep + h % rep) * HEAD_DIM + dc;
    if (v.out_dtype == TWKV_F32) reinterpret_cast<float*>(out)[oi] = val;
    else if (v.out_dtype == TWKV_BF16) reinterpret_cast<unsigned short*>(out)[oi] = from_f32<true>(val);
    else reinterpret_cast<unsigned short*>(out)[oi] = from_f32<false>(val);
  }
  tc::cluster_sync_all();                              // the partners have read this CTA's part
}

// ------------------------------------------------------------------------- host side
cudaError_t launch_kscore_tc(const DevView& v, int layer, const CUtensorMap& map_blocks, const CUtensorMap& map_uinvT,
                             const void* q, int n_pieces, bool pairs, cudaStream_t st);
cudaError_t launch_vacc_tc(const DevView& v, int layer, const CUtensorMap& map_blocks, const CUtensorMap* map_scores, const int* seq_ids,
                           int n_seq, int n_splits, cudaStream_t st);

template <bool BF16>
static cudaError_t launch_decode_t(const DevView& v, int layer, const LayerParams& lp, const void* q, const int* seq_ids,
                                   int n_seq, void* out, int n_splits, int sm_count, const TcMaps* maps, bool pairs, cudaStream_t st) {
  // the K-score kernel's work is cut into one piece per persistent CTA, or per CTA pair
  const int n_pieces = pairs ? kscore_max_pairs(sm_count) : sm_count;
  // CTAs per sequence that invert the V -> K links: enough of them that they finish inside the K work list's time
  const int vj = n_seq >= 256 ? 1 : (256 / n_seq > 64 ? 64 : 256 / n_seq);
  { ProfScope ps(TWKV_K_PLAN, st); plan_kernel<<<1 + n_seq + n_seq * vj, 1024, 0, st>>>(v, layer, seq_ids, n_seq, n_pieces, pairs ? 1 : 0, n_splits, vj); }
  {
    cudaError_t e = launch_kscore_tc(v, layer, maps->blocks, maps->uinvT_k, q, n_pieces, pairs, st);
    if (e != cudaSuccess) return e;
  }
  {
    ProfScope ps(TWKV_K_VACC, st);
    cudaError_t e = launch_vacc_tc(v, layer, maps->blocks, maps->scores, seq_ids, n_seq, n_splits, st);
    if (e != cudaSuccess) return e;
  }
  {
    ProfScope ps(TWKV_K_MERGE, st);
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(MG_THREADS);
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = MG_CL; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const unsigned short* uv = reinterpret_cast<const unsigned short*>(lp.Uinv_v);
    const int wide = (n_seq * v.rep + MW_ROWS - 1) / MW_ROWS;
    cudaError_t e;
    if (MG_CL * wide * v.Hkv >= 2 * sm_count) {
      // 32 rows per cluster while that still makes two CTAs per SM
      cfg.gridDim = dim3(MG_CL * wide, v.Hkv);
      cfg.dynamicSmemBytes = MW_SMEM;
      e = cudaFuncSetAttribute(merge_wide_kernel<BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize, MW_SMEM);
      if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, merge_wide_kernel<BF16>, v, uv, n_splits, n_seq, out);
    } else {
      // query heads per cluster: the whole group, fewer (a divisor) while there are less than two CTAs per SM; then query
      // slots per cluster (they share the reads of U_V^-1) while there are more
      int hp = v.rep, ns = 1;
      while (hp % 2 == 0 && MG_CL * n_seq * v.Hkv * (v.rep / hp) < 2 * sm_count) hp /= 2;
      while (2 * ns * hp <= MG_ROWS && MG_CL * (n_seq * v.Hkv * (v.rep / hp) / (2 * ns)) >= 2 * sm_count) ns *= 2;
      cfg.gridDim = dim3(MG_CL * ((n_seq + ns - 1) / ns), v.Hkv * (v.rep / hp));
      e = cudaLaunchKernelEx(&cfg, merge_kernel<BF16>, v, uv, n_splits, hp, ns, n_seq, out);
    }
    if (e != cudaSuccess) return e;
  }
  count_launch(4);
  return cudaGetLastError();
}

cudaError_t launch_decode(const DevView& v, int layer, const LayerParams& lp, const void* q, const int* seq_ids,
                          int n_seq, void* out, int num_splits, int sm_count, const TcMaps* maps, bool pairs, cudaStream_t st) {
  if (n_seq <= 0) return cudaSuccess;
  return v.dtype == TWKV_BF16 ? launch_decode_t<true>(v, layer, lp, q, seq_ids, n_seq, out, num_splits, sm_count, maps, pairs, st)
                              : launch_decode_t<false>(v, layer, lp, q, seq_ids, n_seq, out, num_splits, sm_count, maps, pairs, st);
}

}  // namespace twkv

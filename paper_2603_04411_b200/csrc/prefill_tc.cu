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
// Precision: as in decode attention, keys are carried as two f16 (21 bits), queries as f16, softmax weights as two parts of
// the cache type; values are two parts of the cache type as well (22 bits for f16, 16 for bf16), so that the result is the
// spectral-space one to rounding.  The products high.high, high.low and low.high of weights and values are formed.
//
// Cost per 128 x 128 tile of (query row, token): 2 + 3 tensor-core units of 2 x 128^3 flop; the softmax of one tile runs
// beside the products of the other.
#include "twkv_dev.h"
#include "tc_util.cuh"
#include "scan_util.cuh"
#include "prefill.h"

namespace twkv {
using namespace tc;

// ------------------------------------------------------------------------------------------ tables
// Zeroes the position bitmaps and maps sequence ids to the call's sequence slots.
__global__ void __launch_bounds__(1024) pf_init_kernel(DevView v, PfCall a) {
  for (int i = blockIdx.x * 1024 + threadIdx.x; i < a.n_words; i += gridDim.x * 1024) a.bits[i] = 0u;
  if (blockIdx.x > 0) return;
  for (int s = threadIdx.x; s < v.S; s += 1024) a.slot[s] = -1;
  __syncthreads();
  for (int u = threadIdx.x; u < a.n_u; u += 1024) { a.slot[a.seqs[3 * u]] = u; a.dup[u] = 0; }
  if (threadIdx.x == 0) *a.ticket = 0;
}

// Sets the bit of every visible token's position; a position met twice marks its sequence.
__global__ void __launch_bounds__(1024) pf_bits_kernel(DevView v, PfCall a, int layer) {
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
}

__device__ __forceinline__ int pf_rank(const PfCall& a, int off, int pos) {      // visible tokens before position pos
  const int w = off + (pos >> 5);
  return a.pref[w] + __popc(a.bits[w] & ((1u << (pos & 31)) - 1u));
}

// Dense row of every K and V slot, position of every row, the segments a tile touches; per query and per block of queries
// what it may see.  The last `qctas` CTAs take the queries.
__global__ void __launch_bounds__(1024) pf_rows_kernel(DevView v, PfCall a, int layer, int qctas) {
  const int tctas = (int)gridDim.x - qctas;
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


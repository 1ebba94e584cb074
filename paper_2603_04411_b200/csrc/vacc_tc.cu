// V-side of decode attention on the 5th-generation tensor cores.
//
// By linearity of Eq. 3 the weighted sum of the values is taken in spectral space: per (query slot, split, head group)
//   acc[j][h] = sum over the split's tokens t of  X^_V[t][j] * p[t][h],   p = exp(s - max) as two parts of the cache dtype,
//   l[h]      = sum over t of p[t][h],
// and merge_kernel projects acc / l through U_V^-1 once.  A V tile of rank class c is c panels [128 tokens x 64
// columns] in HBM.  Two panels at a time form the A operand of one tcgen05.mma chain (M = 128 spectral columns, N = the
// CTA's heads padded to 16 / 32, K = 16 tokens per instruction, 8 instructions per tile): a panel as TMA lands it
// (rows of 128 bytes, 128-byte swizzle) is exactly the MN-major operand layout, the second panel of the pair being the
// second 64-column atom along M (leading byte offset = one panel).  The fp32 accumulator of panel pair i is N columns of
// TMEM (two parts each) at column 2 i N and stays there for the whole kernel; no accumulator lives in registers and the panels are read
// from shared memory by the tensor core only.  A class with an odd number of panels ends with a lone panel; its chain
// points the second atom at a small zero block instead (the leading byte offset is free per instruction), so the pair's
// upper accumulator half adds zeros.
// The probabilities are the B operand (K-major: [head][token], two 64-token halves), written by 8 warps: thread =
// (head, 8 consecutive tokens), one 16-byte swizzled store per 8 weights.  The K-score kernel stores a token's scores at
// its V slot, so a tile's 128 score rows lie next to each other: one TMA box [128 rows x the CTA's heads] per tile,
// issued by the producer thread two tiles ahead into a ring of three tiles in shared memory (TS = true).  A narrow tile
// reads as many bytes of scores as of values, and with one tile in flight their latency bound the kernel.  Where the
// head count is not a multiple of four (rows not 16-byte aligned: no tensor map) each warp copies the rows of its own
// token groups with cp.async instead (TS = false).
// Of a tile that is at most half full (each class of a sequence ends with a partly full one) only the boxes of sixteen rows that hold
// tokens are read, and the products run over as many tokens: a batch of short sequences is bound by the bytes of such tiles.
// Weights go in as two parts of the cache type (see below): 2 N rows of one B operand, so that a panel is read once for both;
// the two halves of the accumulator are added at the end.
//
// Warp roles (320 threads, one CTA per SM):
//   warp 0      TMA producer of V panels (ring of 32-KiB pair stages; one elected lane)
//   warp 1      MMA issuer (one elected lane; owns the TMEM allocation)
//   warps 2-9   probabilities, then at the end the read-out of the accumulators to the split's partial result
// All waits are bounded (tc_util.cuh); a wait that runs out ends the kernel with TWKV_ERR_TIMEOUT.
#include "twkv_dev.h"
#include "tc_util.cuh"
#include "mma_util.cuh"

namespace twkv {
using namespace tc;

constexpr int VT_PWARPS = 8;
constexpr int VT_PTHREADS = 32 * VT_PWARPS;
constexpr int VT_THREADS = 64 + VT_PTHREADS;
constexpr int VT_META = 256;                                   // tiles whose descriptors are staged in shared memory at a time
constexpr uint32_t VT_PANEL_BYTES = 16384;
constexpr uint32_t VT_STAGE_BYTES = 2 * VT_PANEL_BYTES;
constexpr uint32_t VT_ZERO_BYTES = 2048;                       // 16 token rows of zeros: the missing partner of a lone panel
constexpr uint32_t VT_SMEM_MAX = 232448;
constexpr int VT_SC = 3;                                       // tiles of scores in flight (a fourth would cost a stage of the panel ring)

template <bool BF16, int N>
struct VtCfg {
  static constexpr int PARTS = 2;                              // operands per weight (high and low part)
  static constexpr int NB = PARTS * N;                         // rows of the B operand: the N heads' high parts, then their low parts
  static constexpr uint32_t P_PART_BYTES = N * 128;            // [N heads][64 tokens]
  static constexpr uint32_t P_HALF_BYTES = PARTS * P_PART_BYTES;
  static constexpr uint32_t P_BUF_BYTES = 2 * P_HALF_BYTES;
  static constexpr uint32_t TAIL_BYTES = VT_META * 16 + VT_PTHREADS * 4 + 256;      // descriptors, row sums, barriers
  static constexpr uint32_t SC_STAGE_BYTES = 128 * N * 4;      // [128 tokens][N heads] fp32
  static constexpr uint32_t FIXED_BYTES = VT_ZERO_BYTES + 2 * P_BUF_BYTES + VT_SC * SC_STAGE_BYTES + TAIL_BYTES + 1024;   // + alignment slack
  static constexpr int STAGES_FIT = (int)((VT_SMEM_MAX - FIXED_BYTES) / VT_STAGE_BYTES);
  static constexpr int STAGES = STAGES_FIT < 6 ? STAGES_FIT : 6;
  static constexpr uint32_t SMEM_BYTES = STAGES * VT_STAGE_BYTES + FIXED_BYTES;
  static constexpr int ITEMS = N / 16;                         // (head, 8-token group) items per probability thread and tile
};

constexpr float VT_LOG2E = 1.44269504088896340736f;
__device__ __forceinline__ uint64_t vt_pack(float a, float b) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ void vt_unpack(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t vt_fma2(uint64_t a, uint64_t b, uint64_t c) { uint64_t r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ uint64_t vt_add2(uint64_t a, uint64_t b) { uint64_t r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ float vt_ex2(float x) { float r; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x)); return r; }
// Instruction descriptor: kind::f16, fp32 accumulate, A MN-major (bit 15), B K-major, M = 128.
__host__ __device__ constexpr uint32_t vt_idesc(int fmt, int n) { return idesc_f16(fmt, 128, n) | (1u << 15); }

template <bool BF16, int N, bool TS>
__global__ void __launch_bounds__(VT_THREADS, 1)
vacc_tc_kernel(const __grid_constant__ CUtensorMap map_blocks, const __grid_constant__ CUtensorMap map_boxes,
               const __grid_constant__ CUtensorMap map_scores, const __grid_constant__ CUtensorMap map_score_boxes, DevView v,
               const int* seq_ids, int n_splits) {
  chain_start();
  using C = VtCfg<BF16, N>;
  constexpr int S = C::STAGES, ITEMS = C::ITEMS;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int Hq = v.Hq, d_kv = v.d_kv;
  const int qs = blockIdx.x / n_splits, split = blockIdx.x - qs * n_splits;
  const int h0 = blockIdx.y * N, nh = min(N, Hq - h0);
  const int NB = min(N, Hq);                                    // heads per score row in shared memory (TS: the box's width)
  // shared memory: ring | zero block | probabilities [2 buffers][2 halves][2 N][128 B] | score ring | descriptors | row sums | barriers
  const uint32_t s0 = smem_addr(smem_raw);
  const uint32_t pad = (1024u - (s0 & 1023u)) & 1023u;          // operand tiles need 1024-byte alignment for the swizzle
  unsigned char* base_ptr = smem_raw + pad;
  const uint32_t sRing = s0 + pad;
  const uint32_t sZero = sRing + S * VT_STAGE_BYTES;
  const uint32_t sP = sZero + VT_ZERO_BYTES;
  unsigned char* sP_ptr = base_ptr + S * VT_STAGE_BYTES + VT_ZERO_BYTES;
  unsigned char* sS_ptr = sP_ptr + 2 * C::P_BUF_BYTES;                                // score ring
  const uint32_t sS = sP + 2 * C::P_BUF_BYTES;
  int4* s_meta = reinterpret_cast<int4*>(sS_ptr + VT_SC * C::SC_STAGE_BYTES);          // (tile, class, tokens, first block)
  float* s_l = reinterpret_cast<float*>(s_meta + VT_META);
  unsigned char* tail = reinterpret_cast<unsigned char*>(s_l + VT_PTHREADS);
  const uint32_t bars = smem_addr(tail);
  const uint32_t full = bars, empty = full + 8 * S, p_full = empty + 8 * S, p_empty = p_full + 16, acc_done = p_empty + 16;
  const uint32_t sc_full = acc_done + 8, sc_empty = sc_full + 8 * VT_SC;
  uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(tail + 8 * (2 * S + 5 + 2 * VT_SC));
  volatile int* abort_flag = reinterpret_cast<int*>(s_tmem_base + 1);

  const int n_pairs = (v.NC + 1) >> 1;
  uint32_t tmem_cols = 32;
  while (tmem_cols < (uint32_t)(n_pairs * C::NB)) tmem_cols <<= 1;

  if (tid == 0) {
    for (int i = 0; i < S; ++i) { mbar_init(full + 8 * i, 1); mbar_init(empty + 8 * i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(p_full + 8 * i, VT_PWARPS); mbar_init(p_empty + 8 * i, 1); }
    mbar_init(acc_done, 1);
    for (int i = 0; i < VT_SC; ++i) { mbar_init(sc_full + 8 * i, 1); mbar_init(sc_empty + 8 * i, VT_PWARPS); }
    *abort_flag = 0;
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc(smem_addr(s_tmem_base), tmem_cols);
  for (int i = tid; i < (int)VT_ZERO_BYTES / 16; i += VT_THREADS)
    reinterpret_cast<uint4*>(base_ptr + S * VT_STAGE_BYTES)[i] = make_uint4(0u, 0u, 0u, 0u);
  fence_proxy_async_smem();
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem_base = *s_tmem_base;

  chain_wait();
  const int seq = seq_ids[qs];
  const bool seq_ok = seq >= 0 && seq < v.S;
  // this split's range of the sequence's V tiles in stride order, laid out and cut to equal cost by plan_kernel; an id outside
  // the cache has no tiles and contributes nothing: zero partials.  (Walking the cache's own list here took two more dependent reads and
  // the search for the stride: 2 us at the start of every CTA, 4 with 270 tiles per sequence, instead of 1.)
  const int* cut = v.vcut + (size_t)qs * (n_splits + 1) + split;
  const int t_first = cut[0], n_mine = seq_ok ? cut[1] - t_first : 0;
  const int4* meta = v.vmeta + (size_t)(seq_ok ? seq : 0) * v.TPS + t_first;

  // role state that survives the descriptor chunks
  uint32_t st = 0, st_ph = 0;                                   // producer / issuer: ring stage and its phase
  uint32_t n_loaded = 0;                                        // producer: stages filled so far
  uint32_t n_boxes = 0;                                         // producer: score boxes requested so far
  uint32_t touched = 0;                                         // issuer: panel pairs whose accumulator holds a value
  bool ok = true;
  int max_cls = 0;                                              // probability warps: widest class seen (which accumulators to read)
  uint64_t l_sum2 = 0;                                          // probability threads: two sums of this thread's weights

  // probability threads: fixed head, items = 8-token groups
  const int pt = tid - 64;                                      // 0 .. 255 for warps 2-9
  const int ph_ = pt & (N - 1);                                 // head within the CTA's group
  uint64_t nm2 = 0;                                             // minus the head's maximum, in powers of two
  const uint64_t log2e2 = vt_pack(VT_LOG2E, VT_LOG2E);
  if (warp >= 2) {
    // a query that sees no token (chunked prefill, every cached position after its own) has no maximum: weights stay 0
    const float m = ph_ < nh ? dec_ordered(v.seqmax[qs * Hq + h0 + ph_]) : 0.f;
    const float m_h = m == -INFINITY ? 0.f : m;
    nm2 = vt_pack(-m_h * VT_LOG2E, -m_h * VT_LOG2E);
  }

  for (int c0 = 0; c0 < n_mine; c0 += VT_META) {
    const int cn = min(VT_META, n_mine - c0);
    // descriptors of this chunk of the split's tiles
    for (int i = tid; i < cn; i += VT_THREADS) s_meta[i] = meta[c0 + i];
    __syncthreads();

    if (warp == 0) {
      // ------------------------------------------------------------- TMA producer
      if (elect_one()) {
        if (c0 == 0) { tma_prefetch_desc(&map_blocks); if constexpr (TS) tma_prefetch_desc(&map_scores); }
        // the score rows of tile i of the chunk: one box [128 rows x NB heads] into stage (c0 + i) % VT_SC
        auto score_box = [&](int i) -> bool {
          const uint32_t k = (uint32_t)(c0 + i), stg = k % VT_SC;
          if (!mbar_wait_thin(sc_empty + 8 * stg, ((k / VT_SC) & 1u) ^ 1u, abort_flag)) return false;
          const int nb = vtile_boxes(s_meta[i].z), row = s_meta[i].x * TILE;
          mbar_expect_tx(sc_full + 8 * stg, (uint32_t)(nb * JOINT_ROWS * NB * 4));
          if (nb == TILE / JOINT_ROWS) tma_load_2d(sS + stg * C::SC_STAGE_BYTES, &map_scores, sc_full + 8 * stg, h0, row);
          else
            for (int b = 0; b < nb; ++b)
              tma_load_2d(sS + stg * C::SC_STAGE_BYTES + b * JOINT_ROWS * NB * 4, &map_score_boxes, sc_full + 8 * stg, h0, row + b * JOINT_ROWS);
          n_boxes = k + 1;
          return true;
        };
        if constexpr (TS) {
          for (int i = 0; i < 2 && i < cn && ok; ++i) ok = score_box(i);
        }
        for (int i = 0; i < cn && ok; ++i) {
          const int4 m = s_meta[i];
          const int nb = vtile_boxes(m.z);
          if constexpr (TS) {
            if (i + 2 < cn && !(ok = score_box(i + 2))) break;
          }
          for (int j = 0; j < m.y; j += 2) {
            if (!(ok = mbar_wait_thin(empty + 8 * st, st_ph ^ 1u, abort_flag))) break;
            const bool two = j + 1 < m.y;
            if (nb == TILE / JOINT_ROWS) {
              mbar_expect_tx(full + 8 * st, two ? VT_STAGE_BYTES : VT_PANEL_BYTES);
              tma_load_2d(sRing + st * VT_STAGE_BYTES, &map_blocks, full + 8 * st, 0, (m.w + j) * TILE);
              if (two) tma_load_2d(sRing + st * VT_STAGE_BYTES + VT_PANEL_BYTES, &map_blocks, full + 8 * st, 0, (m.w + j + 1) * TILE);
            } else {                                            // only the rows that hold tokens: the products go no further either
              mbar_expect_tx(full + 8 * st, (uint32_t)((two ? 2 : 1) * nb * JOINT_ROWS * PANEL * 2));
              for (int b = 0; b < nb; ++b) {
                const uint32_t dst = sRing + st * VT_STAGE_BYTES + b * (JOINT_ROWS * PANEL * 2);
                tma_load_2d(dst, &map_boxes, full + 8 * st, 0, (m.w + j) * TILE + b * JOINT_ROWS);
                if (two) tma_load_2d(dst + VT_PANEL_BYTES, &map_boxes, full + 8 * st, 0, (m.w + j + 1) * TILE + b * JOINT_ROWS);
              }
            }
            ++n_loaded;
            if (++st == (uint32_t)S) { st = 0; st_ph ^= 1u; }
          }
        }
        if (!ok) {                                              // let copies in flight land before the CTA goes away
          for (uint32_t i = 0; i < (uint32_t)S && i < n_loaded; ++i) {
            const uint32_t n = n_loaded - 1 - i;
            mbar_wait_drain(full + 8 * (n % S), (n / S) & 1u);
          }
          for (uint32_t i = 0; i < (uint32_t)VT_SC && i < n_boxes; ++i) {
            const uint32_t n = n_boxes - 1 - i;
            mbar_wait_drain(sc_full + 8 * (n % VT_SC), (n / VT_SC) & 1u);
          }
        }
      }
      __syncwarp();
    } else if (warp == 1) {
      // ------------------------------------------------------------- MMA issuer
      if (elect_one()) {
        constexpr uint32_t idesc = vt_idesc(BF16 ? 1 : 0, C::NB);
        for (int i = 0; i < cn && ok; ++i) {
          const int k = c0 + i;
          const int cls = s_meta[i].y, nb = vtile_boxes(s_meta[i].z);
          const uint32_t buf = (uint32_t)k & 1u;
          if (!(ok = mbar_wait_thin(p_full + 8 * buf, ((uint32_t)k >> 1) & 1u, abort_flag))) break;
          const uint32_t pb = sP + buf * C::P_BUF_BYTES;
          for (int j = 0; j < cls; j += 2) {
            if (!(ok = mbar_wait_thin(full + 8 * st, st_ph, abort_flag))) break;
            fence_after_sync();
            const uint32_t a0 = sRing + st * VT_STAGE_BYTES;
            const bool two = j + 1 < cls;
            const uint32_t pair = (uint32_t)j >> 1, d_tmem = tmem_base + pair * C::NB;
            uint32_t acc = (touched >> pair) & 1u;
            auto step = [&](int ks) {
              const uint32_t a_addr = a0 + ks * 2048u;                                     // 16 token rows per instruction
              const uint32_t lbo = two ? VT_PANEL_BYTES : sZero - a_addr;                 // where the second 64 columns are
              const uint32_t a_lo = ((a_addr >> 4) & 0x3fffu) | ((lbo >> 4) << 16);
              const uint32_t b_lo = kmajor_sw128_desc_lo(pb + (ks >> 2) * C::P_HALF_BYTES + (ks & 3) * 32u);
              const uint64_t ad = ((uint64_t)KMAJOR_SW128_DESC_HI << 32) | a_lo, bd = ((uint64_t)KMAJOR_SW128_DESC_HI << 32) | b_lo;
              mma_f16_ss(d_tmem, ad, bd, idesc, acc);
              acc = 1u;
            };
            if (nb == TILE / JOINT_ROWS) {                      // (a loop of its own: the checks would cost this thread its pace)
#pragma unroll
              for (int ks = 0; ks < 8; ++ks) step(ks);
            } else {
#pragma unroll 1
              for (int ks = 0; ks < nb; ++ks) step(ks);
            }
            touched |= 1u << pair;
            mma_commit(empty + 8 * st);
            if (++st == (uint32_t)S) { st = 0; st_ph ^= 1u; }
          }
          if (!ok) break;
          mma_commit(p_empty + 8 * buf);
        }
        if (ok && c0 + cn == n_mine) mma_commit(acc_done);
      }
      __syncwarp();
    } else {
      // ------------------------------------------------------------- probabilities
      // One cp.async group per iteration: the score rows of tile i + VT_SC - 1.  Waiting for all but the newest
      // VT_SC - 1 groups then guarantees tile i's scores.  A warp copies and reads only the rows of its own token groups.
      constexpr int GL = N == 16 ? 16 : 32;                     // lanes that share an item
      const int gl = lane & (GL - 1);
      const bool al16 = (Hq & 3) == 0;                          // score rows start on 16-byte boundaries
      // Starts the copies of tile i's score rows into its stage of the score ring.  Every row of the stage is written:
      // rows past the tile's last token, and heads past the CTA's last, get -inf (weight 0).
      auto issue_scores = [&](int i) {
        if (i < cn) {
          const uint32_t stage = (uint32_t)((c0 + i) % VT_SC) * C::SC_STAGE_BYTES;
          const int4 m = s_meta[i];
          const int n_valid = m.z;
          const float* rows = v.scores + (size_t)m.x * TILE * Hq + h0;            // the tile's first score row, at this CTA's heads
          if (al16) {
            constexpr int CPR = N / 4, R = 8 * CPR / GL;        // 16-byte pieces per row; pieces per lane and item
#pragma unroll
            for (int it = 0; it < ITEMS; ++it)
#pragma unroll
              for (int r = 0; r < R; ++r) {
                const int row = ((it * VT_PTHREADS + pt) / N) * 8 + (r * GL + gl) / CPR, ch = (r * GL + gl) % CPR;
                const uint32_t off = stage + (uint32_t)((row * N + 4 * ch) * 4);
                if (row < n_valid && 4 * ch < nh) cp_async16(sS + off, rows + (size_t)row * Hq + 4 * ch);
                else *reinterpret_cast<float4*>(sS_ptr + off) = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
              }
          } else {
            constexpr int R = 8 * N / GL;
#pragma unroll
            for (int it = 0; it < ITEMS; ++it)
#pragma unroll
              for (int r = 0; r < R; ++r) {
                const int row = ((it * VT_PTHREADS + pt) / N) * 8 + (r * GL + gl) / N, hh = (r * GL + gl) % N;
                const uint32_t off = stage + (uint32_t)((row * N + hh) * 4);
                if (row < n_valid && hh < nh) cp_async4(sS + off, rows + (size_t)row * Hq + hh);
                else *reinterpret_cast<float*>(sS_ptr + off) = -INFINITY;
              }
          }
        }
      };
      if constexpr (!TS) {
#pragma unroll 1
        for (int d = 0; d < VT_SC - 1; ++d) { issue_scores(d); cp_async_commit(); }
      }
      for (int i = 0; i < cn && ok; ++i) {
        const int k = c0 + i;
        max_cls = max(max_cls, s_meta[i].y);
        const int n_valid_i = s_meta[i].z;
        if constexpr (TS) {
          if (!(ok = __all_sync(0xffffffffu, mbar_wait(sc_full + 8 * ((uint32_t)k % VT_SC), ((uint32_t)k / VT_SC) & 1u, abort_flag)))) break;
        } else {
          issue_scores(i + VT_SC - 1);
          cp_async_commit();
          cp_async_wait<VT_SC - 1>();                           // this thread's copies of tile i have landed
          __syncwarp();                                         // ... and the other lanes'
        }
        const uint32_t buf = (uint32_t)k & 1u;
        if (!(ok = __all_sync(0xffffffffu, mbar_wait(p_empty + 8 * buf, (((uint32_t)k >> 1) & 1u) ^ 1u, abort_flag)))) break;
        unsigned char* pb = sP_ptr + buf * C::P_BUF_BYTES;
        const float* srow = reinterpret_cast<const float*>(sS_ptr + (uint32_t)(k % VT_SC) * C::SC_STAGE_BYTES) + ph_;
        const int rs = TS ? NB : N;                             // floats per score row in the stage
        // a box holds whatever the scratch holds in rows past the tile's last token and has no columns past the last head
        const bool head_ok = !TS || ph_ < nh, all_valid = n_valid_i == TILE && nh == N;
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
          const int tg = (it * VT_PTHREADS + pt) / N;
          if (tg * 8 >= vtile_boxes(n_valid_i) * JOINT_ROWS) break;      // the products leave these rows out
          // Two weights at a time, packed: exp2 of one fused multiply-add, then the nearest value of the type and the rest.  bf16 keeps 8 bits of a weight, f16 11: with few tokens per sequence that rounding alone reaches 1e-3
          // and 1e-4 of the output, so the remainder goes into a second operand (16 and 22 bits in all).
          // Measured with both parts in one B operand: 64 heads bf16 over 131072 tokens 33.4 us (41.3 with two chains of products and
          // rounded parts), f16 16 x 32768 66.1 us and 64 x 8192 78 us (68.1 and 77.1 with one f16 part).
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int u = 0; u < 8; u += 2) {
            float a0, a1;
            vt_unpack(vt_fma2(vt_pack(srow[(tg * 8 + u) * rs], srow[(tg * 8 + u + 1) * rs]), log2e2, nm2), a0, a1);
            float p0 = vt_ex2(a0), p1 = vt_ex2(a1);
            if (TS && !all_valid) {                             // uniform: tiles with fewer than 128 tokens, CTAs with fewer heads than N
              p0 = (head_ok && tg * 8 + u < n_valid_i) ? p0 : 0.f;
              p1 = (head_ok && tg * 8 + u + 1 < n_valid_i) ? p1 : 0.f;
            }
            const uint64_t p = vt_pack(p0, p1);
            l_sum2 = vt_add2(l_sum2, p);
            split_pair_16<BF16>(p, hi[u >> 1], lo[u >> 1]);
          }
          const uint32_t off = (uint32_t)(tg >> 3) * C::P_HALF_BYTES + (uint32_t)ph_ * 128u + ((((uint32_t)tg & 7u) ^ ((uint32_t)ph_ & 7u)) << 4);
          *reinterpret_cast<uint4*>(pb + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          *reinterpret_cast<uint4*>(pb + C::P_PART_BYTES + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
        fence_proxy_async_smem();
        __syncwarp();                                           // also: the stage is read before the next copies into it start
        if (lane == 0) {
          mbar_arrive(p_full + 8 * buf);
          if constexpr (TS) mbar_arrive(sc_empty + 8 * ((uint32_t)k % VT_SC));
        }
      }
      if constexpr (!TS) cp_async_wait<0>();
    }
    __syncthreads();                                            // the descriptors may be replaced
    ok = ok && !*abort_flag;
  }

  // ----------------------------------------------------------------- partial results of this split
  const size_t pidx = (size_t)qs * n_splits + split;
  if (warp >= 2) {
    {
      float a, b;
      vt_unpack(l_sum2, a, b);
      s_l[pt] = a + b;
    }
    bool ready = ok;
    if (ready && n_mine > 0) ready = __all_sync(0xffffffffu, mbar_wait(acc_done, 0u, abort_flag));
    fence_after_sync();
    float* pa = v.part_acc + (pidx * Hq + h0) * d_kv;
    const int quad = warp & 3;                                  // the TMEM lanes this warp may read
    const int used_pairs = ready ? (max_cls + 1) >> 1 : 0;
    // Sixteen heads at a time through the ring's memory (no copy or product uses it any more) as rows of d_kv floats, from where one
    // bulk copy takes them: consecutive lines in order.  Stored from the registers, sixteen rows 4 KiB apart at a time, the 128 KiB of a
    // CTA took 5.7 us instead of 3.4 (a decode call of 4 x 1000 tokens 51.0 -> 48.4 us, 8 x 5000 82.8 -> 80.4, 37 x 700 143.5 -> 141.0).
    // (a split without tiles leaves its part unwritten: the merge kernel knows it from the cut points)
    float* s_out = reinterpret_cast<float*>(base_ptr);
    for (int n0 = 0; n0 < nh && n_mine > 0; n0 += 16) {
#pragma unroll 1
      for (int pair = (warp - 2) >> 2; pair < n_pairs; pair += 2) {
        const int col = pair * 128 + quad * 32 + lane;          // spectral column of this thread's TMEM lane
        const uint32_t src = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(pair * C::NB);
        float val[16];
        if (pair < used_pairs) {
          float low[16];
          tmem_ld16(src + n0, reinterpret_cast<uint32_t*>(val));
          tmem_ld16(src + N + n0, reinterpret_cast<uint32_t*>(low));
          tmem_ld_wait();
#pragma unroll
          for (int n = 0; n < 16; ++n) val[n] += low[n];
        } else {
#pragma unroll
          for (int n = 0; n < 16; ++n) val[n] = 0.f;
        }
        float* dst = s_out + n0 * d_kv + col;
#pragma unroll
        for (int n = 0; n < 16; ++n) dst[n * d_kv] = val[n];
      }
      fence_proxy_async_smem();
      named_bar_sync(1, VT_PTHREADS);
      if (warp == 2 && elect_one()) bulk_store(pa + (size_t)n0 * d_kv, sRing + (uint32_t)(n0 * d_kv) * 4u, (uint32_t)(min(16, nh - n0) * d_kv) * 4u);
    }
    if (warp == 2 && elect_one()) bulk_store_wait();
    __syncwarp();
    tmem_ld_wait();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  if (warp == 1) tmem_dealloc(tmem_base, tmem_cols);
  if (tid < nh) {
    // row sums: this head's probability threads in index order
    float l = 0.f;
    for (int i = tid; i < VT_PTHREADS; i += N) l += s_l[i];
    v.part_l[pidx * Hq + h0 + tid] = l;
  }
  if (tid == 0 && *abort_flag) set_status(v, TWKV_ERR_TIMEOUT);
}

template <bool BF16, int N, bool TS>
static cudaError_t launch_vacc_tc_n(const DevView& v, const TcMaps& maps, const int* seq_ids, int n_seq, int n_splits, cudaStream_t st) {
  using C = VtCfg<BF16, N>;
  static_assert(C::STAGES >= 3, "the ring needs a few stages");
  static_assert(C::STAGES * VT_STAGE_BYTES >= (uint32_t)N * TWKV_MAX_CLASSES * PANEL * 4, "the partial sums leave through the ring's memory");
  static_assert(C::SMEM_BYTES > CHAIN_TMEM_SMEM, "no other CTA with tensor memory beside this one");
  cudaError_t e = cudaFuncSetAttribute(vacc_tc_kernel<BF16, N, TS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const dim3 grid(n_seq * n_splits, (v.Hq + N - 1) / N);
  e = launch_chained(vacc_tc_kernel<BF16, N, TS>, grid, dim3(VT_THREADS), dim3(1), C::SMEM_BYTES, st, maps.blocks, maps.boxes, TS ? *maps.scores : maps.blocks,
                     TS ? *maps.score_boxes : maps.boxes, v, seq_ids, n_splits);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// maps.scores: the score scratch as a tensor map (boxes of 128 rows x min(N, Hq) heads), or null: rows copied with cp.async.
cudaError_t launch_vacc_tc(const DevView& v, const TcMaps& maps, const int* seq_ids, int n_seq, int n_splits, cudaStream_t st) {
  const bool bf16 = v.dtype == TWKV_BF16;
  // up to 32 heads per CTA; more heads run as further CTAs that read the same panels (through L2)
#define TWKV_VT(BF, NN)                                                                                                   \
  (maps.scores ? launch_vacc_tc_n<BF, NN, true>(v, maps, seq_ids, n_seq, n_splits, st) : launch_vacc_tc_n<BF, NN, false>(v, maps, seq_ids, n_seq, n_splits, st))
  if (v.Hq <= 16) return bf16 ? TWKV_VT(true, 16) : TWKV_VT(false, 16);
  return bf16 ? TWKV_VT(true, 32) : TWKV_VT(false, 32);
#undef TWKV_VT
}

}  // namespace twkv

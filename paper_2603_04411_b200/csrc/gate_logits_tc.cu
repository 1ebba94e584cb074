// Gate logits of Eq. 5 for calls of middle size, and for the soft gate from 128 tokens on: Z = X~ W + b on the 5th-generation tensor
// cores, fp32 logits to the gate scratch, from where the rank kernel of the small calls or the soft gate's kernel takes them.
//
// The fused gate kernel keeps a token's whole row of logits on one CTA pair and leaves most SMs idle in a call of a few token
// tiles; the warp-MMA kernel of the small calls is bound by its own issue from a few hundred tokens on.  With an output tile of
// 128 x 128 per item 1024 tokens of d_kv 1024 fill 128 SMs, and the logits' way through L2 (8 KB per token, both sides) costs less
// than the idle SMs did: a compress call of 1024 tokens takes 46.3 us (warp-MMA 67.6, fused 61.8).  A short call is bound by its
// chain of launches and the latency of one item (16 K panels through the ring).  A ring stage is one K = 64 panel of the states
// (K-major) and of the weights, whose rows are read as the caller's matrix has them (MN-major: two atoms of [64 rows][64 columns]),
// so that the logits are those of the weights at the time of the call and a first call needs no copies of them.
// Warp roles (320 threads): 0 TMA producer, 1 MMA issuer, 2-9 epilogue (thread = one token row x half of the columns).
// All waits are bounded (tc_util.cuh); a wait that runs out ends the kernel with TWKV_ERR_TIMEOUT.
#include "twkv_dev.h"
#include "tc_util.cuh"

namespace twkv {
using namespace tc;

constexpr int GL_THREADS = 320;
constexpr int GL_STAGES = 6;
constexpr uint32_t GL_PANEL_BYTES = 16384, GL_ATOM_BYTES = GL_PANEL_BYTES / 2, GL_STAGE_BYTES = 2 * GL_PANEL_BYTES;
constexpr uint32_t GL_SMEM = GL_STAGES * GL_STAGE_BYTES + 8 * (2 * GL_STAGES + 4) + 16;
static_assert(GL_SMEM > CHAIN_TMEM_SMEM, "no other CTA with tensor memory beside this one");

__global__ void __launch_bounds__(GL_THREADS, 1)
gate_logits_tc_kernel(const __grid_constant__ CUtensorMap map_xk, const __grid_constant__ CUtensorMap map_xv,
                      const __grid_constant__ CUtensorMap map_wk, const __grid_constant__ CUtensorMap map_wv, const float* bias_k,
                      const float* bias_v, int n_tok, int d, int bf16, float* Z, int* status) {
  chain_start();
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int KP = d / PANEL, n_slabs = d / 128;
  const uint32_t sA = smem_addr(smem_raw);
  const bool misaligned = (sA & 1023u) != 0;
  unsigned char* tail = smem_raw + GL_STAGES * GL_STAGE_BYTES;
  const uint32_t bars = smem_addr(tail);
  const uint32_t full = bars, empty = full + 8 * GL_STAGES, acc_full = empty + 8 * GL_STAGES, acc_empty = acc_full + 16;
  uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(tail + 8 * (2 * GL_STAGES + 4));
  volatile int* abort_flag = reinterpret_cast<int*>(s_tmem_base + 1);
  if (tid == 0) {
    for (int i = 0; i < GL_STAGES; ++i) { mbar_init(full + 8 * i, 1); mbar_init(empty + 8 * i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(acc_full + 8 * i, 1); mbar_init(acc_empty + 8 * i, 8); }
    *abort_flag = misaligned ? 1 : 0;
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc(smem_addr(s_tmem_base), 512);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem_base = *s_tmem_base;
  chain_wait();

  // item -> (token tile, side, slab): slab fastest, then side, so that neighbouring CTAs read the same tokens
  const int per_tile = 2 * n_slabs, n_items = per_tile * ((n_tok + TILE - 1) / TILE), it0 = blockIdx.x, itstep = gridDim.x;

  if (misaligned) {
    // nothing was started
  } else if (warp == 0) {
    if (elect_one()) {
      uint32_t st = 0, ph = 0, n_loaded = 0;
      bool ok = true;
      for (int it = it0; it < n_items && ok; it += itstep) {
        const int rem = it % per_tile, m0 = (it / per_tile) * TILE, n0 = (rem % n_slabs) * 128;
        const CUtensorMap *mx = rem >= n_slabs ? &map_xv : &map_xk, *mw = rem >= n_slabs ? &map_wv : &map_wk;
        for (int p = 0; p < KP; ++p, ++n_loaded) {
          if (!(ok = mbar_wait_thin(empty + 8 * st, ph ^ 1u, abort_flag))) break;
          const uint32_t dst = sA + st * GL_STAGE_BYTES;
          mbar_expect_tx(full + 8 * st, GL_STAGE_BYTES);
          tma_load_2d(dst, mx, full + 8 * st, p * PANEL, m0);
          tma_load_2d(dst + GL_PANEL_BYTES, mw, full + 8 * st, n0, p * PANEL);
          tma_load_2d(dst + GL_PANEL_BYTES + GL_ATOM_BYTES, mw, full + 8 * st, n0 + 64, p * PANEL);
          if (++st == GL_STAGES) { st = 0; ph ^= 1u; }
        }
      }
      if (!ok)                                                  // let copies in flight land before the CTA goes away
        for (uint32_t i = 0; i < GL_STAGES && i < n_loaded; ++i) {
          const uint32_t n = n_loaded - 1 - i;
          mbar_wait_drain(full + 8 * (n % GL_STAGES), (n / GL_STAGES) & 1u);
        }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (elect_one()) {
      const uint32_t idesc = idesc_f16(bf16 ? 1 : 0, 128, 128) | (1u << 16);            // B MN-major
      uint32_t st = 0, ph = 0, ac = 0;
      bool ok = true;
      for (int it = it0; it < n_items && ok; it += itstep, ++ac) {
        const uint32_t buf = ac & 1u;
        if (!(ok = mbar_wait(acc_empty + 8 * buf, ((ac >> 1) & 1u) ^ 1u, abort_flag))) break;
        fence_after_sync();
        for (int p = 0; p < KP; ++p) {
          if (!(ok = mbar_wait(full + 8 * st, ph, abort_flag))) break;
          fence_after_sync();
          const uint32_t a_lo = kmajor_sw128_desc_lo(sA + st * GL_STAGE_BYTES), sb = sA + st * GL_STAGE_BYTES + GL_PANEL_BYTES;
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {
            const uint32_t b_lo = (((sb + ks * 2048u) >> 4) & 0x3fffu) | ((GL_ATOM_BYTES >> 4) << 16);
            mma_f16_ss(tmem_base + buf * 256, ((uint64_t)KMAJOR_SW128_DESC_HI << 32) | (a_lo + 2 * ks), ((uint64_t)KMAJOR_SW128_DESC_HI << 32) | b_lo,
                       idesc, (p > 0 || ks > 0) ? 1u : 0u);
          }
          mma_commit(empty + 8 * st);
          if (++st == GL_STAGES) { st = 0; ph ^= 1u; }
        }
        if (ok) mma_commit(acc_full + 8 * buf);
      }
    }
    __syncwarp();
  } else {
    const int quarter = warp & 3, half = (warp - 2) >> 2, row = quarter * 32 + lane;
    const uint32_t src0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + half * 64;
    uint32_t ac = 0;
    for (int it = it0; it < n_items; it += itstep, ++ac) {
      const int rem = it % per_tile, side = rem >= n_slabs, n0 = (rem % n_slabs) * 128 + half * 64;
      const int tok = (it / per_tile) * TILE + row;
      const float* bias = side ? bias_v : bias_k;
      const uint32_t buf = ac & 1u;
      if (!__all_sync(0xffffffffu, mbar_wait(acc_full + 8 * buf, (ac >> 1) & 1u, abort_flag))) break;
      fence_after_sync();
      float x[64];
      tmem_ld32(src0 + buf * 256, reinterpret_cast<uint32_t*>(x));
      tmem_ld32(src0 + buf * 256 + 32, reinterpret_cast<uint32_t*>(x + 32));
      tmem_ld_wait();
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty + 8 * buf);
      if (tok < n_tok) {
        float4* z = reinterpret_cast<float4*>(Z + ((size_t)tok * 2 + side) * d + n0);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const float4 b = bias ? *reinterpret_cast<const float4*>(bias + n0 + 4 * k) : make_float4(0.f, 0.f, 0.f, 0.f);
          z[k] = make_float4(x[4 * k] + b.x, x[4 * k + 1] + b.y, x[4 * k + 2] + b.z, x[4 * k + 3] + b.w);
        }
      }
    }
    tmem_ld_wait();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  if (warp == 1) tmem_dealloc(tmem_base, 512);
  if (tid == 0 && *abort_flag) atomicCAS(status, 0, misaligned ? TWKV_ERR_DEVICE_CHECK : TWKV_ERR_TIMEOUT);
}

// maps: states with boxes of 128 tokens, weights as the caller has them with boxes of 64 rows.
cudaError_t launch_gate_logits_tc(const DevView& v, const GateMaps& maps, const LayerParams& lp, int n_tok, int sm_count, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(gate_logits_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GL_SMEM);
  if (e != cudaSuccess) return e;
  const int items = (n_tok + TILE - 1) / TILE * 2 * (v.d_kv / 128);
  ProfScope ps(TWKV_K_GATE_GEMM, st);
  e = launch_chained(gate_logits_tc_kernel, dim3(items < sm_count ? items : sm_count), dim3(GL_THREADS), dim3(1), GL_SMEM, st, maps.xk, maps.xv, maps.wk,
                     maps.wv, lp.b_k, lp.b_v, n_tok, v.d_kv, v.dtype == TWKV_BF16 ? 1 : 0, v.gate_scratch, v.status);
  count_launch();
  return e;
}

}  // namespace twkv

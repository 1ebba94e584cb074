// Gate logits of Eq. 5: Z = X~ W + b for the K side and the V side (COMPUTE mode).
// A dense contraction [n_tok x d_kv] x [d_kv x d_kv]: 128 x 128 output tiles on the tensor cores,
// 16-bit operands, fp32 accumulation, bias added in the epilogue.
#include "twkv_dev.h"
#include "mma_util.cuh"
#include "tc_util.cuh"

namespace twkv {

// For calls of fewer than 128 tokens (the append of a decode step): one CTA per output tile would leave most SMs idle (16 CTAs), each
// walking all of d_kv with a memory round trip per step, so a cluster of `ks` CTAs shares a tile, a part of d_kv each, and adds the
// partial tiles through distributed shared memory in fixed order (4 tokens: 20.3 -> 12.3 us with cold weights).
constexpr int GG_STAGES = 3;
constexpr int GG_THREADS = 256;

template <bool BF16>
__global__ void __launch_bounds__(GG_THREADS, 1)
gate_gemm_kernel(const unsigned short* Xk, const unsigned short* Xv, const unsigned short* Wk, const unsigned short* Wv, const float* bk,
                 const float* bv, int n_tok, int d, int ks_n, float* Z) {
  chain_start();
  {
    const size_t bytes = (size_t)d * d * 2;
    const unsigned t = ((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * GG_THREADS + threadIdx.x;
    const unsigned n = gridDim.x * gridDim.y * gridDim.z * GG_THREADS;
    l2_prefetch(Wk, bytes, t, n);
    l2_prefetch(Wv, bytes, t, n);
  }
  chain_wait();
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* sA = smem;
  unsigned char* sB = smem + GG_STAGES * 16384;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int side = blockIdx.z / ks_n, kp = blockIdx.z - side * ks_n, m0 = blockIdx.x * 128, n0 = blockIdx.y * 128;
  const unsigned short* X = side ? Xv : Xk;
  const unsigned short* W = side ? Wv : Wk;
  const float* bias = side ? bv : bk;
  const int iters = d / 64 / ks_n, k0 = kp * iters;               // this CTA's part of the contraction, in steps of 64
  auto issue = [&](int it) {
    if (it < iters) {
      const int st = it % GG_STAGES;
      const unsigned dA = smem_u32(sA + st * 16384), dB = smem_u32(sB + st * 16384);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = tid + i * GG_THREADS, row = c >> 3, ch = c & 7;
        const int grow = min(m0 + row, n_tok - 1);            // rows past the end repeat the last row (never stored)
        if (m0 + (row & ~15) < n_tok)                         // sixteen-row groups without a token are not read at all
          cp_async16(dA + row * 128 + ((ch ^ (row & 7)) << 4),
                     reinterpret_cast<const unsigned char*>(X) + ((size_t)grow * d + (k0 + it) * 64) * 2 + ch * 16);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = tid + i * GG_THREADS, kr = c >> 4, ch = c & 15;
        cp_async16(dB + kr * 256 + ((ch ^ (kr & 7)) << 4),
                   reinterpret_cast<const unsigned char*>(W) + ((size_t)((k0 + it) * 64 + kr) * d + n0) * 2 + ch * 16);
      }
    }
    cp_async_commit();
  };
  for (int it = 0; it < GG_STAGES - 1; ++it) issue(it);
  float acc[16][4];
#pragma unroll
  for (int n = 0; n < 16; ++n) { acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f; }
  const int mat = lane >> 3, rin = lane & 7;
  const bool busy = m0 + warp * 16 < n_tok;                       // this warp's rows hold tokens
  for (int it = 0; it < iters; ++it) {
    const int st = it % GG_STAGES;
    cp_async_wait<GG_STAGES - 2>();
    __syncthreads();
    issue(it + GG_STAGES - 1);
    if (!busy) continue;
    const unsigned aBase = smem_u32(sA + st * 16384), bBase = smem_u32(sB + st * 16384);
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      unsigned a[4];
      {
        const int row = warp * 16 + rin + (mat & 1) * 8, kc = ks * 2 + (mat >> 1);
        ldsm_x4(a, aBase + row * 128 + ((kc ^ (row & 7)) << 4));
      }
#pragma unroll
      for (int np = 0; np < 8; ++np) {
        unsigned b[4];
        const int kr = ks * 16 + rin + (mat & 1) * 8, nc = np * 2 + (mat >> 1);
        ldsm_x4_t(b, bBase + kr * 256 + ((nc ^ (kr & 7)) << 4));
        mma16816<BF16>(acc[np * 2], a, b[0], b[1]);
        mma16816<BF16>(acc[np * 2 + 1], a, b[2], b[3]);
      }
    }
  }
  cp_async_wait<0>();
  if (ks_n > 1) {
    __syncthreads();                                              // the stages become the partial tile [128][128]
    float* part = reinterpret_cast<float*>(smem);
    const int pr = warp * 16 + (lane >> 2);
#pragma unroll
    for (int n = 0; n < 16 && busy; ++n) {
      const int pc = n * 8 + (lane & 3) * 2;
      *reinterpret_cast<float2*>(part + pr * 128 + pc) = make_float2(acc[n][0], acc[n][1]);
      *reinterpret_cast<float2*>(part + (pr + 8) * 128 + pc) = make_float2(acc[n][2], acc[n][3]);
    }
    tc::cluster_sync_all();
    const int rows = min(128, n_tok - m0);
    for (int i = kp * GG_THREADS + tid; i < rows * 32; i += ks_n * GG_THREADS) {       // four columns of one row
      const int r = i >> 5, c = (i & 31) * 4;
      const uint32_t at = tc::smem_addr(part + r * 128 + c);
      float4 s = bias ? *reinterpret_cast<const float4*>(bias + n0 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
      for (int k = 0; k < ks_n; ++k) {
        float4 x;
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(tc::cluster_map(at, k)));
        s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
      }
      *reinterpret_cast<float4*>(Z + ((size_t)(m0 + r) * 2 + side) * d + n0 + c) = s;
    }
    tc::cluster_sync_all();                                       // the partners have read this CTA's part
    return;
  }
  const int r0 = m0 + warp * 16 + (lane >> 2), r1 = r0 + 8;
#pragma unroll
  for (int n = 0; n < 16; ++n) {
    const int col = n0 + n * 8 + (lane & 3) * 2;
    const float b0 = bias ? bias[col] : 0.f, b1 = bias ? bias[col + 1] : 0.f;
    if (r0 < n_tok) *reinterpret_cast<float2*>(Z + ((size_t)r0 * 2 + side) * d + col) = make_float2(acc[n][0] + b0, acc[n][1] + b1);
    if (r1 < n_tok) *reinterpret_cast<float2*>(Z + ((size_t)r1 * 2 + side) * d + col) = make_float2(acc[n][2] + b0, acc[n][3] + b1);
  }
}

cudaError_t launch_gate_logits(const DevView& v, const LayerParams& lp, const void* K, const void* V, int n_tok,
                               float* logits, cudaStream_t st) {
  if (n_tok <= 0) return cudaSuccess;
  const size_t smem = 2 * GG_STAGES * 16384;
  int ks = 8;                                                     // CTAs per tile; d_kv / 64 may be an odd number
  while ((v.d_kv / 64) % ks) ks /= 2;
  ProfScope ps(TWKV_K_GATE_GEMM, st);
  auto X = [](const void* p) { return reinterpret_cast<const unsigned short*>(p); };
  auto kernel = v.dtype == TWKV_BF16 ? gate_gemm_kernel<true> : gate_gemm_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)
    e = launch_chained(kernel, dim3((n_tok + 127) / 128, v.d_kv / 128, 2 * ks), dim3(GG_THREADS), dim3(1, 1, ks), smem, st, X(K), X(V), X(lp.W_k),
                       X(lp.W_v), lp.b_k, lp.b_v, n_tok, v.d_kv, ks, logits);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace twkv

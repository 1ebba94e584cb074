// Global token eviction (the paper's combination with token eviction, Sec. 5.2 "Implementation Details": the spectral
// decomposition is joint across heads, so a token is kept or dropped for all heads at once) and compaction of the
// survivors inside the cache.
//
//   twkv_evict(cache, layer, seq, keep_positions, n_keep): of the tokens cached for `seq` in `layer`, exactly those
//   whose position is listed survive, on the K side and on the V side.
// Container rule.  For every (side, class) of the sequence the survivors move to the front of the tiles that key
// already owns, in their stored order; the vacated rows of the last tile that stays in use are zeroed; tiles left
// without a token are taken off the tile lists (their blocks stay unused until the cache is reset).  V slots are
// relinked to the new slots of their tokens' K rows.  Later appends continue behind the survivors.
//
// Four launches: (1) bitmap of the kept positions; (2) per key, the destination of every slot (nothing moves yet: the
// V side finds a token's position through its K row); (3) per key and panel, the moves (a round's rows are all read before
// any is written, destinations never lie behind sources); (4) the tile lists without the emptied tiles.
#include "twkv_dev.h"
#include "scan_util.cuh"

namespace twkv {

constexpr int EV_THREADS = 1024;

// The tiles of key (side, seq, cls) in creation order -> s_tiles; returns their number.  K tiles are listed per class
// (all sequences), V tiles per sequence (all classes); both lists are in creation order.
__device__ int collect_key_tiles(const DevView& v, int layer, int side, int seq, int cls, int* s_tiles, int* s_warp) {
  const int4* desc = v.desc(layer, side);
  const int* list = side ? v.svt(layer) + (size_t)seq * v.TPS : v.kct(layer) + (size_t)(cls - 1) * v.NT;
  const int n = side ? v.svc(layer)[seq] : v.kcc(layer)[cls - 1];
  int base = 0;
  for (int i0 = 0; i0 < n; i0 += EV_THREADS) {
    const int i = i0 + threadIdx.x;
    int t = -1, mine = 0;
    if (i < n) {
      t = list[i];
      const int4 d = desc[t];
      mine = (d.x == seq && d.y == cls) ? 1 : 0;
    }
    int total;
    const int off = block_scan_excl(mine, s_warp, &total);
    if (mine) s_tiles[base + off] = t;
    base += total;
  }
  __syncthreads();
  return base;
}

__global__ void __launch_bounds__(EV_THREADS) evict_bitmap_kernel(DevView v, int layer, int seq, const int* keep, int n_keep) {
  chain_start();
  chain_wait();
  unsigned* bm = v.evict_bitmap;
  for (int i = threadIdx.x; i < (ROPE_LO * ROPE_HI) / 32; i += EV_THREADS) bm[i] = 0u;
  __syncthreads();
  for (int i = threadIdx.x; i < n_keep; i += EV_THREADS) {
    const int p = keep[i];
    if (p >= 0 && p < ROPE_LO * ROPE_HI) atomicOr(&bm[p >> 5], 1u << (p & 31));
  }
  if (threadIdx.x == 0) v.stok(layer)[seq] = 0;            // the K-side keys add their survivors back
}

// grid (NC, 2): one CTA per key of the sequence.  evict_map[side][tile * 128 + slot] = new global slot, or -1.
__global__ void __launch_bounds__(EV_THREADS) evict_plan_kernel(DevView v, int layer, int seq) {
  chain_start();
  chain_wait();
  extern __shared__ int s_tiles[];
  __shared__ int s_warp[32];
  const int cls = blockIdx.x + 1, side = blockIdx.y, tid = threadIdx.x;
  const int nk = collect_key_tiles(v, layer, side, seq, cls, s_tiles, s_warp);
  const int4* desc = v.desc(layer, side);
  const int* aux = v.aux(layer, side);
  const int* kaux = v.aux(layer, 0);
  const unsigned short* rank = v.rank(layer, side);
  int* map = v.evict_map + (size_t)side * v.NT * TILE;
  int base = 0;
  unsigned long long dropped = 0ull;
  for (int j0 = 0; j0 < nk; j0 += EV_THREADS / TILE) {
    const int j = j0 + tid / TILE, slot = tid % TILE;
    int keep = 0, t = -1;
    if (j < nk) {
      t = s_tiles[j];
      if (slot < desc[t].z) {
        const int a = aux[(size_t)t * TILE + slot];
        const int pos = side ? kaux[a] : a;                // a V slot links to its token's K slot, which holds the position
        keep = (v.evict_bitmap[pos >> 5] >> (pos & 31)) & 1u;
        if (!keep) dropped += rank[(size_t)t * TILE + slot];
      }
    }
    int total;
    const int off = block_scan_excl(keep, s_warp, &total);
    if (t >= 0) {
      const int g = base + off;
      map[(size_t)t * TILE + slot] = keep ? s_tiles[g / TILE] * TILE + g % TILE : -1;
    }
    base += total;
  }
  // dropped ranks leave the layer's rank sums (Eq. 4 statistics)
  for (int o = 16; o > 0; o >>= 1) dropped += __shfl_xor_sync(0xffffffffu, dropped, o);
  if ((tid & 31) == 0 && dropped) atomicAdd(&v.rank_sums[layer * 2 + side], 0ull - dropped);
  if (tid == 0) {
    const int key = (side * v.S + seq) * v.NC + (cls - 1);
    v.evict_fill[side * v.NC + cls - 1] = base;             // the move kernel commits it
    v.key_last_l(layer)[key] = base > 0 ? s_tiles[(base - 1) / TILE] : -1;
    if (side == 0 && base) atomicAdd(&v.stok(layer)[seq], base);
  }
}

// grid (NC, 2, NC): the moves of one panel of one key (panels are separate blocks and move alike; the CTA of panel 0 also moves
// positions / links and ranks and commits the counts).  Source tiles are taken in order, EV_BATCH tiles per round: every row is
// read into registers, the CTA synchronises, then the survivors are written; a destination never lies behind its source, so
// a round overwrites only rows that have been read.  What bounds it is the chain of rounds, one memory round trip each: 8192
// tokens of all classes 41.4 -> 16.9 us against one CTA per key that took its tiles and panels one by one.
constexpr int EV_BATCH = 4;
__global__ void __launch_bounds__(EV_THREADS) evict_move_kernel(DevView v, int layer, int seq) {
  chain_start();
  chain_wait();
  extern __shared__ int s_tiles[];
  __shared__ int s_warp[32];
  const int cls = blockIdx.x + 1, side = blockIdx.y, panel = blockIdx.z, tid = threadIdx.x;
  if (panel >= cls) return;
  const int nk = collect_key_tiles(v, layer, side, seq, cls, s_tiles, s_warp);
  int4* desc = v.desc(layer, side);
  int* aux = v.aux(layer, side);
  unsigned short* rank = v.rank(layer, side);
  const int* map = v.evict_map + (size_t)side * v.NT * TILE;
  const int* kmap = v.evict_map;
  const int new_fill = v.evict_fill[side * v.NC + cls - 1];
  const int slot = tid >> 3;                                // this thread's 16 bytes of a tile's panel: row tid / 8, piece tid % 8
  for (int j0 = 0; j0 < nk; j0 += EV_BATCH) {
    uint4 piece[EV_BATCH];
    unsigned char* dst[EV_BATCH];
#pragma unroll
    for (int b = 0; b < EV_BATCH; ++b) {
      dst[b] = nullptr;
      if (j0 + b < nk) {
        const int t = s_tiles[j0 + b], to = map[(size_t)t * TILE + slot];
        if (to >= 0 && to != t * TILE + slot) {
          piece[b] = *reinterpret_cast<const uint4*>(v.blocks + (size_t)(desc[t].w + panel) * BLOCK_BYTES + slot * 128 + (tid & 7) * 16);
          dst[b] = v.blocks + (size_t)(desc[to / TILE].w + panel) * BLOCK_BYTES + (to % TILE) * 128 + (tid & 7) * 16;
        }
      }
    }
    // positions / links and ranks: thread = (tile of the round, slot)
    int a = 0, to_slot = -1;
    unsigned short r = 0;
    if (panel == 0 && tid < EV_BATCH * TILE && j0 + tid / TILE < nk) {
      const int from = s_tiles[j0 + tid / TILE] * TILE + tid % TILE;
      to_slot = map[from];
      if (to_slot >= 0) {
        a = aux[from];
        if (side) a = kmap[a];                              // the token's K row has moved too
        r = rank[from];
      }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < EV_BATCH; ++b)
      if (dst[b]) *reinterpret_cast<uint4*>(dst[b]) = piece[b];
    if (to_slot >= 0) { aux[to_slot] = a; rank[to_slot] = r; }
    __syncthreads();
  }
  // rows behind the last survivor in the last tile still in use are zero, as after an append
  const int kept = (new_fill + TILE - 1) / TILE;
  if (kept > 0 && new_fill % TILE) {
    const int first = new_fill % TILE;
    uint4* rows = reinterpret_cast<uint4*>(v.blocks + (size_t)(desc[s_tiles[kept - 1]].w + panel) * BLOCK_BYTES + first * 128);
    if (tid < (TILE - first) * 8) rows[tid] = make_uint4(0u, 0u, 0u, 0u);
  }
  if (panel > 0) return;
  for (int j = tid; j < nk; j += EV_THREADS) desc[s_tiles[j]].z = j < kept ? min(TILE, new_fill - j * TILE) : 0;
  if (tid == 0) v.fill_l(layer)[(side * v.S + seq) * v.NC + (cls - 1)] = new_fill;
}

// grid NC + 1: the K tile list of every class, and the sequence's V tile list, without the emptied tiles of `seq`
__global__ void __launch_bounds__(EV_THREADS) evict_lists_kernel(DevView v, int layer, int seq) {
  chain_start();
  chain_wait();
  __shared__ int s_warp[32];
  const bool vlist = (int)blockIdx.x == v.NC;
  const int side = vlist ? 1 : 0;
  const int4* desc = v.desc(layer, side);
  int* list = vlist ? v.svt(layer) + (size_t)seq * v.TPS : v.kct(layer) + (size_t)blockIdx.x * v.NT;
  int* count = vlist ? v.svc(layer) + seq : v.kcc(layer) + blockIdx.x;
  const int n = *count;
  int base = 0;
  for (int i0 = 0; i0 < n; i0 += EV_THREADS) {
    const int i = i0 + threadIdx.x;
    int t = -1, stay = 0;
    if (i < n) {
      t = list[i];
      const int4 d = desc[t];
      stay = (d.x == seq && d.z == 0) ? 0 : 1;
    }
    int total;
    const int off = block_scan_excl(stay, s_warp, &total);   // (its barriers also separate this round's reads from the writes)
    if (stay) list[base + off] = t;
    base += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) *count = base;
}

cudaError_t launch_evict(const DevView& v, int layer, int seq, const int* keep_positions, int n_keep, cudaStream_t st) {
  const size_t smem = (size_t)v.TPS * sizeof(int);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(evict_plan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(evict_move_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  ProfScope ps(TWKV_K_OTHER, st);
  const dim3 b(EV_THREADS), one(1);
  cudaError_t e = launch_chained(evict_bitmap_kernel, one, b, one, 0, st, v, layer, seq, keep_positions, n_keep);
  if (e == cudaSuccess) e = launch_chained(evict_plan_kernel, dim3(v.NC, 2), b, one, smem, st, v, layer, seq);
  if (e == cudaSuccess) e = launch_chained(evict_move_kernel, dim3(v.NC, 2, v.NC), b, one, smem, st, v, layer, seq);
  if (e == cudaSuccess) e = launch_chained(evict_lists_kernel, dim3(v.NC + 1), b, one, 0, st, v, layer, seq);
  if (e != cudaSuccess) return e;
  count_launch(4);
  return cudaGetLastError();
}

}  // namespace twkv

// Decode attention over the mixed-rank cache (Eq. 3, reshape to heads, RoPE, softmax attention).
//
//   plan_kernel    running-max reset, K-tile work list; cut points of every
//                  sequence's V tiles into the splits of the V pass; K slot -> V slot links of the sequences' tokens
//   kscore_tc_kernel (kscore_tc.cu)  per K tile: Kbar = X^_K U_K^-1, RoPE by stored position,
//                  s = q . Kbar * scale for the GQA group, scores to scratch, per-sequence max
//   vacc_tc_kernel (vacc_tc.cu)  per (sequence, split): p = exp(s - max), acc += p^T X^_V in spectral
//                  space (tcgen05), l = sum p
//   merge_kernel   sum of the splits, out_h = (acc_h / l_h) U_V^-1[:, head slice]
//
// V is never reconstructed per token: by linearity of Eq. 3 the weighted sum is taken in
// spectral space and projected once.
#include <algorithm>

#include "twkv_dev.h"
#include "mma_util.cuh"
#include "tc_util.cuh"
#include "scan_util.cuh"

namespace twkv {

// ------------------------------------------------------------------------------ plan
// One launch prepares a decode pass.  CTAs 0 .. NC-1, one per rank class: the class's part of the K-score work list, the K
// tiles of the listed sequences in table order, classes one behind the other from wide to narrow; for the CTA-pair kernel as
// items of two tiles of one class.  Where a class's part starts follows from the keys' token counts (a key of n tokens has
// ceil(n / 128) tiles), so the classes need not wait for one another; a class is compacted by block-wide scans, so the order
// does not depend on thread timing.  CTA 0 also cuts the list into n_cta contiguous pieces of about equal estimated cost, so
// that a CTA (pair) of the K-score kernel mostly stays inside one (class, sequence) run.  What bounds it is the chain of
// dependent table reads: one CTA that walked the whole list took 17.5 us for 16 sequences of 32768 tokens (2200 tiles) and 17
// for 64 of 8192; a CTA per class took 8.6 and 9.5 (8.9 -> 8.4 for 8 tiles).  The tables of the joint tiles (below) have CTAs of
// their own, and a class's first tiles are asked for before anything is counted.
// cycles per tile of the K-score kernel by rank class: a least-squares fit, one coefficient per class, of every CTA's busy
// time to its tile counts on the benchmark's mix of classes (8 KV heads, CTA pairs; residual 1.3 us rms of 330): a fixed
// part (rotation factors, the per-slab epilogue and score products) plus a per-panel part, an odd panel count costing a
// little more than the even one above it saves; classes above 8 run as two passes.  Only the ratios matter.
__constant__ unsigned kTileCost[TWKV_MAX_CLASSES] = {14300u, 16600u, 18600u, 19500u, 22100u, 23000u, 25400u, 26200u,
                                                   38800u, 38700u, 42000u, 42800u, 45600u, 45800u, 49300u, 50700u};
__device__ __forceinline__ unsigned ktile_cost(int cls) { return kTileCost[min(max(cls, 1), TWKV_MAX_CLASSES) - 1]; }

// Cut points of one sequence's V tile list into n_splits contiguous ranges of about equal cost (a tile costs its
// panels' rows that hold tokens plus its score rows, counted in 512-byte units): the V pass is bound by the bytes a CTA reads, and tiles of
// classes 1 to 16 dealt out by count alone left the slowest CTA with half as much again as the mean.
// The list is taken in the stride order of vtile_stride(); cut[s] = number of tiles (in that order) whose inclusive cost
// prefix is <= s / n_splits of the total; split s takes positions cut[s] .. cut[s + 1] - 1 of that order.
// min_splits > 0: the caller left the number open.  A sequence then uses that many, or one per DECODE_SPLIT_TOKENS of its tokens; the
// rest stay empty.  Decided here, from what the cache holds when the call runs, and not on the host, a replayed call splits as an
// eager one does.
__device__ void vsplit_plan(const DevView& v, int layer, const int* seq_ids, int qs, int n_splits, int min_splits) {
  __shared__ int s_warp[32];
  const int tid = threadIdx.x;
  const int seq = seq_ids[qs];
  const int n = (seq >= 0 && seq < v.S) ? v.svc(layer)[seq] : 0;
  const int* list = v.svt(layer) + (size_t)(n > 0 ? seq : 0) * v.TPS;
  const int4* desc = v.desc(layer, 1);
  int* cut = v.vcut + (size_t)qs * (n_splits + 1);
  const int stride = vtile_stride(n);
  int4* meta = v.vmeta + (size_t)(n > 0 ? seq : 0) * v.TPS;
  // cost of the i-th tile in stride order (its sum over a list stays below 2^31: 32 * 16 + 64 units, at most 2^13 tiles), whose
  // description the V pass finds in that order
  auto cost = [&](int i) -> int {
    if (i >= n) return 0;
    const int t = list[vtile_at(i, stride, n)];
    const int4 d = desc[t];
    meta[i] = make_int4(t, d.y, d.z, d.w);
    return TILE / 32 * vtile_boxes(d.z) * d.y + v.Hq;
  };
  // a list of up to 1024 tiles is read once; a longer one first for its total
  const int first = cost(tid);
  int total = 0, w = first, off = 0;
  for (int i0 = 0; i0 < n; i0 += 1024) {
    int part;
    off = block_scan_excl(i0 ? cost(i0 + tid) : w, s_warp, &part);
    total += part;
  }
  if (total == 0) {
    for (int s = tid; s <= n_splits; s += 1024) cut[s] = 0;
    return;
  }
  const int used = min_splits > 0 ? min(n_splits, max(min_splits, v.stok(layer)[seq] / DECODE_SPLIT_TOKENS)) : n_splits;
  const unsigned long long W = (unsigned long long)total, ns = (unsigned long long)used;
  int base = 0;
  for (int i0 = 0; i0 < n; i0 += 1024) {
    if (n > 1024) {
      int part;
      w = i0 ? cost(i0 + tid) : first;
      off = base + block_scan_excl(w, s_warp, &part);
      base += part;
    }
    if (i0 + tid < n) {
      const unsigned long long e = (unsigned long long)off, p = e + (unsigned long long)w;
      // the splits whose boundary floor(s W / ns) falls in [e, p): they start at this tile
      for (unsigned long long s = (e * ns + W - 1ull) / W; s < ns && s * W / ns < p; ++s) cut[s] = i0 + tid;
    }
  }
  if (used + tid <= n_splits) cut[used + tid] = n;               // (the library's own choice is at most 64)
}

// Joint tiles.  A key (sequence, class) ends with a tile that is partly full, and sixteen of those cost a short sequence several times
// its tokens: the K-score kernel pays for a tile, not for its rows.  The last tiles of a sequence are therefore laid together, from the
// widest class to the narrowest, as long as their rows (rounded up to boxes of sixteen) fit one tile; it has the class of its first, and
// the narrower ones' missing panels are zeros.  Every row is computed as in a tile of its own, so the scores are the same bit for bit.
// A decode call in us, a tile per class / joint tiles: 16 x 500 82.7 / 60.5, 64 x 1000 216 / 146, 37 x 700 of any rank 140 / 105,
// 32 x 2000 139 / 111, 4 x 1000 44.7 / 41.7, 8 x 5000 74.3 / 72.2; long sequences, whose tiles are nearly all full, pay for the tables:
// 1 x 30000 62.4 / 64.6, 4 x 8192 61.0 / 62.7.
// Returns the classes (bit class - 1) at which a joint tile starts, and << 16 the classes that lie in one.
__device__ unsigned joint_masks(const DevView& v, int layer, int seq) {
  const int* fill = v.fill_l(layer) + (size_t)seq * v.NC;
  int boxes[TWKV_MAX_CLASSES];
#pragma unroll
  for (int k = 0; k < TWKV_MAX_CLASSES; ++k) boxes[k] = k < v.NC ? ((fill[k] & (TILE - 1)) + JOINT_ROWS - 1) / JOINT_ROWS : 0;
  unsigned starts = 0u, joined = 0u, run = 0u, first = 0u;       // of the run being laid together: its classes, the widest
  int used = 0;
#pragma unroll
  for (int k = TWKV_MAX_CLASSES - 1; k >= 0; --k) {
    const int b = boxes[k];
    if (b == 0 || b == TILE / JOINT_ROWS) continue;
    if (used + b > TILE / JOINT_ROWS) {
      if (run != first) { starts |= first; joined |= run; }
      run = 0u; used = 0;
    }
    if (run == 0u) first = 1u << k;
    run |= 1u << k;
    used += b;
  }
  if (run != first) { starts |= first; joined |= run; }
  return starts | (joined << 16);
}

// One warp writes the tables of the joint tile of sequence `seq` that starts at class index k0 (bit k0 of the masks).
__device__ void joint_tile(const DevView& v, int layer, int seq, unsigned masks, int k0, int id) {
  const int lane = threadIdx.x & 31;
  const unsigned below = masks & ((1u << k0) - 1u);               // the next joint tile's first class, if any, ends this one
  unsigned members = (masks >> 16) & ((2u << k0) - 1u);
  if (below) members &= ~((2u << (31 - __clz(below))) - 1u);
  const bool in = lane < TWKV_MAX_CLASSES && ((members >> lane) & 1u);
  const int key = seq * v.NC + lane;
  const int rest = in ? v.fill_l(layer)[key] & (TILE - 1) : 0, tile = in ? v.key_last_l(layer)[key] : 0;
  const int block = in ? v.desc(layer, 0)[tile].w : 0, room = (rest + JOINT_ROWS - 1) / JOINT_ROWS * JOINT_ROWS;
  int at = room;                                                  // wide classes first: the rooms of the lanes above
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_down_sync(0xffffffffu, at, o);
    if (lane + o < 32) at += u;
  }
  at -= room;
  int slot[4] = {-1, -1, -1, -1};
  unsigned box = 0u;
  for (unsigned m = members; m; m &= m - 1) {
    const int k = __ffs(m) - 1;
    const int a = __shfl_sync(0xffffffffu, at, k), n = __shfl_sync(0xffffffffu, rest, k), rm = __shfl_sync(0xffffffffu, room, k);
    const int t = __shfl_sync(0xffffffffu, tile, k), b = __shfl_sync(0xffffffffu, block, k);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = 32 * j + lane - a;
      if (r >= 0 && r < n) slot[j] = t * TILE + r;
    }
    const int r = JOINT_ROWS * lane - a;
    if (r >= 0 && r < rm) box = (unsigned)((b * TILE + r) / JOINT_ROWS) << 5 | (unsigned)(k + 1);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    v.joint_rows()[(size_t)id * TILE + 32 * j + lane] = slot[j];
    v.joint_pos()[(size_t)id * TILE + 32 * j + lane] = slot[j] >= 0 ? v.aux(layer, 0)[slot[j]] : 0;
  }
  if (lane < TILE / JOINT_ROWS) v.joint_boxes()[(size_t)id * (TILE / JOINT_ROWS) + lane] = box;
}

// K slot -> V slot of every token of one sequence (the V slots carry the opposite link): the K-score kernel stores a
// token's scores at its V slot, so that the V pass finds a tile's score rows next to each other.  CTA j of the vj CTAs of
// a sequence takes the V tiles j * 8 .. j * 8 + 7, then vj * 8 further on, eight tiles (1024 slots) at a time.
__device__ void vlink_plan(const DevView& v, int layer, const int* seq_ids, int qs, int j, int vj) {
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

__global__ void __launch_bounds__(1024) plan_kernel(DevView v, int layer, const int* seq_ids, int n_seq, int n_cta, int pairs,
                                                    int n_splits, int min_splits, int vj, const void* uinv_k, const void* uinv_v) {
  chain_start();
  {
    const size_t bytes = (size_t)v.d_kv * v.d_kv * 2;             // the bases, which the K pass and the merge read (32 layers in turn find them
    // in HBM: 4 sequences of 1000 tokens, append and decode, 101.5 -> 100.8 us per layer with this and the gate's prefetch)
    const unsigned t = blockIdx.x * 1024 + threadIdx.x, n = gridDim.x * 1024;
    l2_prefetch(uinv_k, bytes, t, n);
    l2_prefetch(uinv_v, bytes, t, n);
  }
  chain_wait();
  const int NC = v.NC;
  if ((int)blockIdx.x >= NC + 2 * n_seq) {                        // the last n_seq * vj CTAs: K slot -> V slot links
    const int idx = (int)blockIdx.x - NC - 2 * n_seq;
    vlink_plan(v, layer, seq_ids, idx / vj, idx % vj, vj);
    return;
  }
  if ((int)blockIdx.x >= NC + n_seq) {                            // before them n_seq CTAs: the tables of a sequence's joint tiles, a warp each
    const int i = (int)blockIdx.x - NC - n_seq, seq = seq_ids[i];
    if (threadIdx.x >= TWKV_MAX_CLASSES / 2 * 32 || seq < 0 || seq >= v.S) return;
    const unsigned masks = joint_masks(v, layer, seq);
    unsigned starts = masks & 0xffffu;
    for (int w = threadIdx.x >> 5; w > 0 && starts; --w) starts ^= 1u << (31 - __clz(starts));
    if (starts) joint_tile(v, layer, seq, masks, 31 - __clz(starts), i * (NC / 2) + (threadIdx.x >> 5));
    return;
  }
  if ((int)blockIdx.x >= NC) {                                    // before those n_seq CTAs: the V pass's split plan, one sequence each
    vsplit_plan(v, layer, seq_ids, (int)blockIdx.x - NC, n_splits, min_splits);
    return;
  }
  extern __shared__ int s_slot[];                                 // sequence id -> query slot, -1; behind it, per query slot, its joint tiles
  unsigned* s_joint = reinterpret_cast<unsigned*>(s_slot + v.S);
  __shared__ int s_warp[32];
  __shared__ int s_keep[TWKV_MAX_CLASSES];                        // tiles of the listed sequences per class
  __shared__ int s_any[TWKV_MAX_CLASSES];                         // whether joint tiles start at the class
  __shared__ int s_koff[TWKV_MAX_CLASSES + 1], s_ioff[TWKV_MAX_CLASSES + 1];    // start of run k (class NC - k) in the tile list / in the item list
  __shared__ unsigned long long s_coff[TWKV_MAX_CLASSES + 1];     // estimated cost of everything before run k
  __shared__ int s_hg;                                            // parts per item
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int run = blockIdx.x, cls = NC - run;
  // the class's first 1024 tiles are asked for at once: they arrive while the joint tiles and the counts are worked out
  const int n_list = v.kcc(layer)[cls - 1];
  const int4* desc = v.desc(layer, 0);
  const int* list = v.kct(layer) + (size_t)(cls - 1) * v.NT;
  const int t_first = tid < n_list ? list[tid] : 0;
  const int4 d_first = tid < n_list ? desc[t_first] : make_int4(0, 0, 0, 0);
  for (int s = tid; s < v.S; s += 1024) s_slot[s] = -1;
  if (tid < TWKV_MAX_CLASSES) s_keep[tid] = s_any[tid] = 0;
  __syncthreads();
  for (int i = tid; i < n_seq; i += 1024) {
    const int s = seq_ids[i];
    unsigned joint = 0u;
    if (s >= 0 && s < v.S) {
      s_slot[s] = i;
      joint = joint_masks(v, layer, s);
    }
    s_joint[i] = joint;
  }
  for (int i = run * 1024 + tid; i < n_seq * v.Hq; i += NC * 1024) v.seqmax[i] = 0u;
  __syncthreads();
  // (an id outside the cache, or listed again later, has no tiles here)
  auto listed = [&](int i) -> int { const int s = seq_ids[i]; return s >= 0 && s < v.S && s_slot[s] == i ? s : -1; };
  for (int i = tid; i < n_seq; i += 1024) {
    if (listed(i) >= 0) continue;
    s_joint[i] = 0u;
    if (run == 0) set_status(v, TWKV_ERR_INVALID_ARG);                                 // also a duplicate id
  }
  __syncthreads();
  {
    // tiles per class: a warp per class (and part of the sequences), a lane per sequence
    const int parts = 32 / NC, k = warp % NC, part = warp / NC;
    int mine = 0;
    if (part < parts)
      for (int i = part * 32 + lane; i < n_seq; i += parts * 32) {
        const int s = listed(i);
        if (s < 0) continue;
        const int f = v.fill_l(layer)[s * NC + k];
        const unsigned j = s_joint[i];
        const int joint = (int)((j >> k) & 1u);
        mine += f / TILE + (f % TILE != 0 && !((j >> (16 + k)) & 1u) ? 1 : 0) + joint;
        if (joint) s_any[k] = 1;
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if (lane == 0 && mine) atomicAdd(&s_keep[k], mine);
  }
  __syncthreads();
  if (warp == 0) {
    // lane k = run k (class NC - k): where its tiles, items and costs start
    const int keep = lane < NC ? s_keep[NC - lane - 1] : 0, items = pairs ? (keep + 1) / 2 : keep;
    int ko = keep, io = items;
    unsigned long long co = (unsigned long long)items * ktile_cost(NC - lane);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int a = __shfl_up_sync(0xffffffffu, ko, o), b = __shfl_up_sync(0xffffffffu, io, o);
      const unsigned long long c = __shfl_up_sync(0xffffffffu, co, o);
      if (lane >= o) { ko += a; io += b; co += c; }
    }
    if (lane < NC) { s_koff[lane + 1] = ko; s_ioff[lane + 1] = io; s_coff[lane + 1] = co; }
    if (lane == 0) { s_koff[0] = s_ioff[0] = 0; s_coff[0] = 0ull; }
    io = __shfl_sync(0xffffffffu, io, 31); co = __shfl_sync(0xffffffffu, co, 31);
    // The KV heads of an item may be dealt out to several CTAs (pairs): finer work for lists that leave some idle or that a few
    // wide tiles decide.  A part repeats the tile's loads and rotation factors.  Least estimate of the slowest piece, in cycles:
    // the widest part where every part has a CTA to itself, else the mean piece plus most of the widest part (numbers fitted to
    // lists of this kind).  A decode call in us, whole items / this rule (ranks 1 .. 512): 1 x 8192 50.6 / 49.4, 4 x 1000 51.1 / 48.8,
    // 8 x 8192 102.6 / 102.4, 16 x 500 62.6 / 63.2; 64 x 2000 and 16 x 32768 keep whole items.
    constexpr float PART_COST = 2600.f;
    const unsigned used = __ballot_sync(0xffffffffu, items > 0);
    const float wide_cost = used ? (float)ktile_cost(NC - (__ffs(used) - 1)) : 0.f, per_cta = 1.f / (float)n_cta;
    float best = 3.4e38f, part = 1.f;
    int parts = 1;
    for (int h = 1; v.Hkv % h == 0; h *= 2, part *= 0.5f) {
      const float est = io * h <= n_cta ? wide_cost * part
                                        : ((float)co + (float)io * (float)(h - 1) * PART_COST) * per_cta + 0.7f * wide_cost * part;
      if (est < best) { best = est; parts = h; }
    }
    if (lane == 0) s_hg = parts;
  }
  __syncthreads();
  // this class's entries; a run of odd length ends with a filler for the pair kernel: the same tile again, flagged so that its
  // scores are dropped
  const int n_keep = s_koff[run + 1] - s_koff[run];
  int base = 0;
  auto put = [&](const int4& e) {                                 // the next entries, of the threads that have one (.w >= 0), in thread order
    int total;
    const int at = base + block_scan_excl(e.w >= 0 ? 1 : 0, s_warp, &total);
    if (e.w >= 0 && at < n_keep) {
      if (pairs) {
        v.kpairs[2 * s_ioff[run] + at] = e;
        if (at == n_keep - 1 && (n_keep & 1)) v.kpairs[2 * s_ioff[run] + at + 1] = make_int4(e.x, e.y | 0x80, e.z, e.w);
      } else {
        v.klist[s_koff[run] + at] = e;
      }
    }
    base += total;
  };
  for (int i0 = 0; i0 < n_list; i0 += 1024) {
    int4 e = make_int4(0, 0, 0, -1);
    if (i0 + tid < n_list) {
      const int t = i0 ? list[i0 + tid] : t_first;
      const int4 d = i0 ? desc[t] : d_first;
      int slot = s_slot[d.x];
      if (slot >= 0 && d.z < TILE && ((s_joint[slot] >> (15 + cls)) & 1u)) slot = -1;     // lies in a joint tile
      e = make_int4(t, d.y | (d.z << 8), d.w, slot);
    }
    put(e);
  }
  // the joint tiles that start at this class; their numbers count the sequence's from the widest on
  for (int i0 = 0; i0 < n_seq && s_any[cls - 1]; i0 += 1024) {
    const int i = i0 + tid;
    const bool mine = i < n_seq && ((s_joint[i] >> (cls - 1)) & 1u);
    put(mine ? make_int4(~(i * (NC / 2) + __popc((s_joint[i] & 0xffffu) >> cls)), cls | (TILE << 8), 0, i) : make_int4(0, 0, 0, -1));
  }
  if (run > 0) return;
  // (the parts the KV heads of an item are dealt out in: chosen above)
  const int n_items = s_ioff[NC], hg = s_hg;
  const unsigned long long total = s_coff[NC];
  if (tid == 0) { *v.kitem_parts = hg; v.cta_start[n_cta] = n_items * hg; }
  // cut points: piece b starts at the item part whose cost interval holds b / n_cta of the total (64-bit arithmetic; inside
  // a run every part costs the same, so the part follows from a division)
  for (int b = tid; b < n_cta; b += 1024) {
    int start = 0;
    if (n_items > 0 && total > 0ull) {
      const unsigned long long key = (unsigned long long)b * total / (unsigned long long)n_cta;
      int k = 0;
      while (k + 1 < NC && s_coff[k + 1] <= key) ++k;
      const unsigned long long within = (key - s_coff[k]) * hg / ktile_cost(NC - k);
      const int cap = (s_ioff[k + 1] - s_ioff[k]) * hg;
      start = s_ioff[k] * hg + (int)(within < (unsigned long long)cap ? within : (unsigned long long)cap);
    }
    v.cta_start[b] = start;
  }
}

// -------------------------------------------------------------- merge + V projection
// A cluster of eight CTAs per (query slots, query heads of one KV head g): ROWS rows (slot, head) at most.  CTA c takes
// the spectral components [c d/8, (c+1) d/8): it sums their splits, normalises, and multiplies by its rows of
// U_V^-1[:, g*128 .. g*128+127]; every CTA hands each of the others its part of 16 columns through distributed shared memory and
// adds the eight parts of its own.  What bounds it is latency: one CTA doing a group's whole sum and product went
// through 256 KiB of U_V^-1 and every split by itself.  Empty splits are not read (the V pass does not write them).
// A cluster of four rows takes 6 us, one of sixteen 15 (its share of the splits, then the FMAs: 67 M of them for 512 rows), so all
// of them are to be resident at once (merge_rows(), below), three CTAs per SM: U_V^-1 waits in shared memory, not in registers.
// 4 sequences of 1000 tokens ran as 512 CTAs in three rounds, 17 us.  A whole call in us, two CTAs per SM / three: 1 x 300
// 40.1 / 36.7, 4 x 1000 48.4 / 44.7, 4 x 8192 65.2 / 61.0, 8 x 5000 80.4 / 74.3, 16 x 500 91.2 / 82.7, 2 x 2000 with 64 heads
// 45.9 / 42.1, 1 x 131072 with 64 heads 145.9 / 140.5; more CTAs than fit and as many rows as fit, two per SM: 4 x 1000 57.0 / 51.0.
constexpr int MG_THREADS = 256;
constexpr int MG_CL = 8;                             // CTAs of a cluster

// shared memory: slice of U_V^-1 [d / 8][128] and, once it has been used, the quarters' products [4][rows][128] | sums | parts | 1 / l
constexpr size_t MG_U_BYTES = 128 * 128 * 2;
__host__ __device__ constexpr size_t merge_acc_bytes(int rows) { return rows * 512 > MG_THREADS * 16 ? rows * 512 : MG_THREADS * 16; }
constexpr size_t merge_smem(int rows) { return MG_U_BYTES + merge_acc_bytes(rows) + rows * 512 + rows * sizeof(float); }

template <bool BF16, int ROWS>
__global__ void __launch_bounds__(MG_THREADS, 3)
merge_kernel(DevView v, const unsigned short* Uinv_v, int n_splits, int hp, int ns, int n_seq, void* out) {
  extern __shared__ __align__(16) unsigned char mg_smem[];
  static_assert(4 * ROWS * 512 <= (int)MG_U_BYTES, "the quarters' products fit where U_V^-1 was");
  const unsigned* s_u = reinterpret_cast<const unsigned*>(mg_smem);                 // pairs of columns
  float* s_red = reinterpret_cast<float*>(mg_smem);
  float* s_acc = reinterpret_cast<float*>(mg_smem + MG_U_BYTES);                     // [rows][d / 8] normalised
  float4* s_part = reinterpret_cast<float4*>(s_acc);                                 // before that: split sums per (split group, row, four components)
  float* s_in = s_acc + merge_acc_bytes(ROWS) / sizeof(float);                       // [CTA of the cluster][row][16 columns of this CTA]
  float* s_invl = s_in + ROWS * 128;
  chain_start();
  tc::cluster_arrive();                              // waited for before the first remote store: the partners run
  chain_wait();
  // blockIdx.y = KV head g and which hp of its query heads; blockIdx.x / 8 = ns query slots that share the reads of U_V^-1
  const int c = tc::cluster_cta_rank();
  const int qs0 = (blockIdx.x / MG_CL) * ns, parts = v.rep / hp, g = blockIdx.y / parts, tid = threadIdx.x, lane = tid & 31;
  const int Hq = v.Hq, d_kv = v.d_kv;
  const int rows = min(ns, n_seq - qs0) * hp;
  const int head0 = g * v.rep + (blockIdx.y % parts) * hp;      // first query head of this CTA
  const int jn = d_kv / MG_CL, j0 = c * jn;                     // jn: a multiple of 16, at most 128
  // row sums over the splits: warp w takes rows w and w + 8, its lanes read the splits' parts together, lane 0 adds them in split
  // order; the first reads go out before everything else
  constexpr int LR = (ROWS + 7) / 8;
  float l_first[LR];
#pragma unroll
  for (int k = 0; k < LR; ++k) {
    const int r = (tid >> 5) + 8 * k;
    l_first[k] = r < rows && lane < n_splits ? v.part_l[((size_t)(qs0 + r / hp) * n_splits + lane) * Hq + head0 + r % hp] : 0.f;
  }
  // this CTA's slice of U_V^-1 does not depend on the sums: on its way meanwhile
  for (int i = tid; i < jn * 16; i += MG_THREADS)
    cp_async16(tc::smem_addr(mg_smem) + i * 16, reinterpret_cast<const uint4*>(Uinv_v + (size_t)(j0 + (i >> 4)) * d_kv + g * HEAD_DIM) + (i & 15));
  cp_async_commit();
  // split sums: a thread owns four components of one row (two rows of sixteen) and every sg_n-th split, with eight reads in flight
  const int q4 = jn / 4, slots = rows * q4, sg_n = slots < MG_THREADS ? MG_THREADS / slots : 1, sg = slots < MG_THREADS ? tid / slots : 0;
  for (int sl = slots < MG_THREADS ? tid - sg * slots : tid; sl < slots && sg < sg_n; sl += MG_THREADS) {
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
        t[k] = s < n_splits && cut[s + 1] > cut[s] ? p[(size_t)s * stride] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) { a.x += t[k].x; a.y += t[k].y; a.z += t[k].z; a.w += t[k].w; }
    }
    s_part[sg * slots + sl] = a;
  }
#pragma unroll
  for (int k = 0; k < LR; ++k) {
    const int r = (tid >> 5) + 8 * k;
    if (r >= rows) break;
    float l = 0.f;
    for (int s0 = 0; s0 < n_splits; s0 += 32) {
      const float mine = s0 == 0 ? l_first[k]
                                 : s0 + lane < n_splits ? v.part_l[((size_t)(qs0 + r / hp) * n_splits + s0 + lane) * Hq + head0 + r % hp] : 0.f;
      const int n = min(32, n_splits - s0);
      for (int s = 0; s < n; ++s) l += __shfl_sync(0xffffffffu, mine, s);
    }
    if (lane == 0) s_invl[r] = l > 0.f ? 1.f / l : 0.f;
  }
  __syncthreads();
  for (int sl = tid; sl < slots; sl += MG_THREADS) {  // in place: nobody else reads or writes these entries
    float4 a = s_part[sl];
    for (int k = 1; k < sg_n; ++k) {                   // fixed order
      const float4 b = s_part[k * slots + sl];
      a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
    }
    const float il = s_invl[sl / q4];
    *reinterpret_cast<float4*>(s_acc + sl * 4) = make_float4(a.x * il, a.y * il, a.z * il, a.w * il);
  }
  cp_async_wait<0>();
  __syncthreads();
  // thread = a pair of columns, a quarter of the components
  const int dp = tid & 63, jg = tid >> 6, jr = jn / 4;
  float o[ROWS][2];
#pragma unroll
  for (int h = 0; h < ROWS; ++h) { o[h][0] = 0.f; o[h][1] = 0.f; }
#pragma unroll 2
  for (int t = 0; t < jr; t += 4) {                    // jr is a multiple of 4
    float u0[4], u1[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const unsigned w = s_u[(jg * jr + t + e) * 64 + dp];
      u0[e] = to_f32<BF16>((unsigned short)(w & 0xffffu)); u1[e] = to_f32<BF16>((unsigned short)(w >> 16));
    }
#pragma unroll
    for (int h = 0; h < ROWS; ++h)
      if (h < rows) {
        const float4 a = *reinterpret_cast<const float4*>(s_acc + h * jn + jg * jr + t);
        o[h][0] += a.x * u0[0]; o[h][1] += a.x * u1[0];
        o[h][0] += a.y * u0[1]; o[h][1] += a.y * u1[1];
        o[h][0] += a.z * u0[2]; o[h][1] += a.z * u1[2];
        o[h][0] += a.w * u0[3]; o[h][1] += a.w * u1[3];
      }
  }
  __syncthreads();                                     // U_V^-1 has been used by everyone
#pragma unroll
  for (int h = 0; h < ROWS; ++h)
    if (h < rows) *reinterpret_cast<float2*>(s_red + (jg * ROWS + h) * 128 + 2 * dp) = make_float2(o[h][0], o[h][1]);
  __syncthreads();
  constexpr int CW = 128 / MG_CL;                      // columns a CTA writes
  tc::cluster_wait();
  for (int i = tid; i < rows * 32; i += MG_THREADS) {  // four columns of a row, to the CTA that writes them
    const int h = i >> 5, c4 = (i & 31) * 4;
    float4 a = *reinterpret_cast<const float4*>(s_red + h * 128 + c4);
#pragma unroll
    for (int k = 1; k < 4; ++k) {
      const float4 b = *reinterpret_cast<const float4*>(s_red + (k * ROWS + h) * 128 + c4);
      a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
    }
    tc::st_cluster_f32x4(tc::cluster_map(tc::smem_addr(s_in + (c * ROWS + h) * CW + c4 % CW), c4 / CW), a);
  }
  tc::cluster_sync_all();                              // every part has arrived; nothing remote is touched from here on
  for (int i = tid; i < rows * CW; i += MG_THREADS) {
    const int h = i / CW, dc = c * CW + i % CW;
    float val = 0.f;
#pragma unroll
    for (int k = 0; k < MG_CL; ++k) val += s_in[(k * ROWS + h) * CW + i % CW];            // fixed order
    const int oslot = qs0 + h / hp;
    const size_t oi = ((size_t)(v.qmap ? v.qmap[oslot] : oslot) * Hq + head0 + h % hp) * HEAD_DIM + dc;
    if (v.out_dtype == TWKV_F32) reinterpret_cast<float*>(out)[oi] = val;
    else if (v.out_dtype == TWKV_BF16) reinterpret_cast<unsigned short*>(out)[oi] = from_f32<true>(val);
    else reinterpret_cast<unsigned short*>(out)[oi] = from_f32<false>(val);
  }
}

__device__ __forceinline__ float ld_cluster_f32(uint32_t addr) {
  float x;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(addr));
  return x;
}

// The same for large batches: 32 rows per cluster share a CTA's slice of U_V^-1, staged in shared memory; thread = (pair of
// columns, a quarter of the rows).  With eight rows the reads of U_V^-1 (256 KiB per eight rows and KV head) bound it:
// 64 sequences of 8192 tokens 63 -> 44.5 us, 37 of up to 700 tokens 42 -> 28 us (43 with one CTA per KV head).
constexpr int MW_ROWS = 32;
constexpr int MW_SMEM = 128 * 128 * 2 + 2 * MW_ROWS * 128 * 4 + MW_ROWS * 4;

template <bool BF16>
__global__ void __launch_bounds__(MG_THREADS)
merge_wide_kernel(DevView v, const unsigned short* Uinv_v, int n_splits, int n_seq, void* out) {
  extern __shared__ __align__(16) unsigned char mw_smem[];
  unsigned* s_u = reinterpret_cast<unsigned*>(mw_smem);                                // [d / 8][64] pairs of columns
  float* s_acc = reinterpret_cast<float*>(mw_smem + 128 * 128 * 2);                    // [rows][d / 8]
  float* s_out = s_acc + MW_ROWS * 128;                                                // [rows][128]
  float* s_invl = s_out + MW_ROWS * 128;
  chain_start();
  chain_wait();
  const int c = tc::cluster_cta_rank(), g = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ns = MW_ROWS / v.rep, qs0 = (blockIdx.x / MG_CL) * ns;
  const int Hq = v.Hq, d_kv = v.d_kv, rep = v.rep;
  const int rows = min(ns, n_seq - qs0) * rep;
  const int jn = d_kv / MG_CL, j0 = c * jn;
  for (int i = tid; i < jn * 16; i += MG_THREADS) {                                    // 16-byte pieces of this CTA's rows of U_V^-1
    const uint4 w = reinterpret_cast<const uint4*>(Uinv_v + (size_t)(j0 + (i >> 4)) * d_kv + g * HEAD_DIM)[i & 15];
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
        t[k] = s0 + k < n_splits && cut[s0 + k + 1] > cut[s0 + k] ? p[(size_t)(s0 + k) * stride] : make_float4(0.f, 0.f, 0.f, 0.f);
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
cudaError_t launch_kscore_tc(const DevView& v, int layer, const CUtensorMap& map_blocks, const CUtensorMap& map_boxes, const CUtensorMap& map_uinvT,
                             const void* q, int n_pieces, bool pairs, cudaStream_t st);
cudaError_t launch_vacc_tc(const DevView& v, const TcMaps& maps, const int* seq_ids,
                           int n_seq, int n_splits, cudaStream_t st);

// Clusters of the merge kernel that are resident at once on the current device, empty (those of sixteen rows, which need the most).
template <bool BF16>
static int merge_clusters_t(int sm_count) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = MG_CL; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(MG_CL); cfg.blockDim = dim3(MG_THREADS); cfg.dynamicSmemBytes = merge_smem(16);
  cfg.attrs = &attr; cfg.numAttrs = 1;
  int n = 0;
  if (cudaFuncSetAttribute(merge_kernel<BF16, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)merge_smem(16)) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, merge_kernel<BF16, 16>, &cfg) != cudaSuccess || n < 1) { cudaGetLastError(); n = sm_count / MG_CL; }
  return n - n / 16;                                     // behind another kernel not quite as many find room together
}
int merge_clusters(bool bf16, int sm_count) { return bf16 ? merge_clusters_t<true>(sm_count) : merge_clusters_t<false>(sm_count); }

// Rows (query slot, query head of a KV head) per cluster of the merge, hp heads of ns slots: as few as still leave all clusters
// resident at once (a second round of clusters starts when the first has ended); query heads of one slot first, then slots.  False
// where sixteen rows are not enough: rows of 32 (merge_wide_kernel).
bool merge_rows(int n_seq, int n_kv_heads, int rep, int fit, int* hp, int* ns) {
  *hp = *ns = 1;
  auto clusters = [&] { return (n_seq + *ns - 1) / *ns * n_kv_heads * (rep / *hp); };
  while (*hp < rep && clusters() > fit) *hp *= 2;
  while (2 * *hp * *ns <= 16 && *ns < n_seq && clusters() > fit) *ns *= 2;
  return clusters() <= fit;
}

template <bool BF16>
static cudaError_t launch_decode_t(const DevView& v, int layer, const LayerParams& lp, const void* q, const int* seq_ids,
                                   int n_seq, void* out, int n_splits, int min_splits, int sm_count, int merge_fit, const TcMaps* maps,
                                   bool pairs, cudaStream_t st) {
  // the K-score kernel's work is cut into one piece per persistent CTA, or per CTA pair
  const int n_pieces = pairs ? kscore_max_pairs(sm_count) : sm_count;
  // CTAs per sequence that invert the V -> K links: enough of them that they finish inside the K work list's time
  const int vj = n_seq >= 128 ? 1 : std::min(64, (256 - n_seq) / n_seq);
  {
    ProfScope ps(TWKV_K_PLAN, st);
    cudaError_t e = launch_chained(plan_kernel, dim3(v.NC + n_seq * (2 + vj)), dim3(1024), dim3(1), (size_t)v.S * 2 * sizeof(int), st, v, layer, seq_ids,
                                   n_seq, n_pieces, pairs ? 1 : 0, n_splits, min_splits, vj, maps->uinv_k, lp.Uinv_v);
    if (e != cudaSuccess) return e;
  }
  {
    cudaError_t e = launch_kscore_tc(v, layer, maps->blocks, maps->boxes, maps->uinvT_k, q, n_pieces, pairs, st);
    if (e != cudaSuccess) return e;
  }
  {
    ProfScope ps(TWKV_K_VACC, st);
    cudaError_t e = launch_vacc_tc(v, *maps, seq_ids, n_seq, n_splits, st);
    if (e != cudaSuccess) return e;
  }
  {
    ProfScope ps(TWKV_K_MERGE, st);
    const unsigned short* uv = reinterpret_cast<const unsigned short*>(lp.Uinv_v);
    const int wide = (n_seq * v.rep + MW_ROWS - 1) / MW_ROWS;
    cudaError_t e;
    int hp, ns;
    if (!merge_rows(n_seq, v.Hkv, v.rep, merge_fit, &hp, &ns)) {
      e = cudaFuncSetAttribute(merge_wide_kernel<BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize, MW_SMEM);
      if (e == cudaSuccess) e = launch_chained(merge_wide_kernel<BF16>, dim3(MG_CL * wide, v.Hkv), dim3(MG_THREADS), dim3(MG_CL), MW_SMEM, st, v, uv, n_splits, n_seq, out);
    } else {
      const dim3 grid(MG_CL * ((n_seq + ns - 1) / ns), v.Hkv * (v.rep / hp));
      auto go = [&](auto kernel, int rows) {
        cudaError_t r = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)merge_smem(rows));
        return r != cudaSuccess ? r : launch_chained(kernel, grid, dim3(MG_THREADS), dim3(MG_CL), merge_smem(rows), st, v, uv, n_splits, hp, ns, n_seq, out);
      };
      e = hp * ns <= 4 ? go(merge_kernel<BF16, 4>, 4) : hp * ns <= 8 ? go(merge_kernel<BF16, 8>, 8) : go(merge_kernel<BF16, 16>, 16);
    }
    if (e != cudaSuccess) return e;
  }
  count_launch(3);                                     // the K-score launch counts itself
  return cudaGetLastError();
}

cudaError_t launch_decode(const DevView& v, int layer, const LayerParams& lp, const void* q, const int* seq_ids,
                          int n_seq, void* out, int num_splits, int min_splits, int sm_count, int merge_fit, const TcMaps* maps, bool pairs, cudaStream_t st) {
  if (n_seq <= 0) return cudaSuccess;
  return v.dtype == TWKV_BF16 ? launch_decode_t<true>(v, layer, lp, q, seq_ids, n_seq, out, num_splits, min_splits, sm_count, merge_fit, maps, pairs, st)
                              : launch_decode_t<false>(v, layer, lp, q, seq_ids, n_seq, out, num_splits, min_splits, sm_count, merge_fit, maps, pairs, st);
}

}  // namespace twkv

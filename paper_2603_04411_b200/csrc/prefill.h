// Tables and buffers of one tiled prefill call (prefill_tc.cu); all of it lies in scratch regions of the cache's pool.
#pragma once
#include <cuda.h>
#include "twkv_dev.h"

namespace twkv {

constexpr int PF_SCALE_MIN = -60;                // of the exponent of the call's values
constexpr int PF_SLOT_FLOATS = 2 * 130 * TILE;    // partial result of (block of queries, KV head, split): [2 tiles][128 output columns, maximum, sum][128 rows]

struct PfCall {
  // the call's queries, sorted by (sequence, position) on the host
  const int* qrow;      // [n] row of q / out
  const int* qpos;      // [n]
  const int2* blocks;   // [n_blocks] (first query, sequence slot << 9 | number of queries): at most two tiles of rows, one sequence
  const int* seqs;      // [n_u][3] sequence id, largest query position, first word of its bitmap
  int n_u, n_blocks, n_words;
  int blk0, blk_n;      // the group of blocks handled now
  int n_splits, seg_rows;
  int seg_rest;         // segments that the positions alone can need; further ones are for repeated positions
  // made on the device
  int* slot;            // [max_seqs] sequence id -> sequence slot of the call, -1
  unsigned* bits;       // [n_words] bitmaps of the visible positions
  int* pref;            // [n_words] set bits before the word, inside the sequence
  int *rows, *base, *dup;   // [n_u] rows of a sequence, its first dense row, whether a position repeats
  int *ticket, *total;      // [1] rows of the call, every sequence's rounded up to whole tiles
  int* qvis;            // [n] rows of its sequence a query may see
  int4* binfo;          // [n_blocks] first dense row of the sequence, most rows a query of the block sees, repeated positions
  int* krow;            // [NT * 128] K-tile-order rows of sequences with a repeated position
  int *krow_out, *vrow; // [NT * 128] dense row of every K / V slot, -1 = not visible
  int* rowpos;          // [rows] position of a dense row
  unsigned char* seg_buf;   // [Hkv][4 parts][seg_rows][128] 16-bit
  const unsigned short* uv; // U_V^-1 of the layer
  float* vscale;        // [2] the power of two the call's values are multiplied by before they are split, and its inverse
  // the power of two a row's value was divided by besides, per KV head; segment + 1 of the last segment
  // in which a block of 128 rows held one other than 0
  signed char* vexp;    // [Hkv][seg_rows]
  int* vflag;           // [seg_rows / 128][Hkv]
  float* slots;         // [blk_n * Hkv * n_splits][PF_SLOT_FLOATS]
};
struct PfMaps { CUtensorMap blocks, uk, uv, seg; };

// out: where one split of one segment is a query's whole result, the attention kernel writes the outputs itself and the combine
// kernel, launched for what may turn out otherwise, leaves
cudaError_t launch_pf_tables(const DevView& v, const PfCall& a, int layer, int sm_count, cudaStream_t st);
cudaError_t launch_pf_segment(const DevView& v, const PfCall& a, const PfMaps& maps, int layer, int seg, const void* q, void* out, int sm_count, cudaStream_t st);
cudaError_t launch_pf_combine(const DevView& v, const PfCall& a, void* out, cudaStream_t st);

}  // namespace twkv

// What the packing paths share (pack.cu: any size; pack_small.cu: one launch for small inputs; pack_split.cu: larger ones).
#pragma once

#include "common.cuh"

namespace comet {

enum { kStatusRange = 0, kStatusDuplicate = 1, kStatusInvalid = 2, kStatusOverflow = 3 };   // words of Context::d_status

struct KeyLayout {
  int order;
  int shift[COMET_MAX_ORDER];      // bit position of level l's coordinate inside the key
  int bits[COMET_MAX_ORDER];
  int total_bits;
  int64_t dim[COMET_MAX_ORDER];    // extent of the mode stored at level l
};

struct CoordPtrs { const int32_t *p[COMET_MAX_ORDER]; };   // level order

// ORDER is a template parameter so that the per-level loops unroll and the by-value descriptor structs
// are read with constant indices (a runtime index would push them into local memory).
template <int ORDER>
__device__ __forceinline__ uint64_t entry_key(const CoordPtrs &c, const KeyLayout &k, int64_t p, bool &bad) {
  int32_t v[ORDER];
#pragma unroll
  for (int l = 0; l < ORDER; ++l) v[l] = __ldcs(c.p[l] + p);
  uint64_t key = 0;
#pragma unroll
  for (int l = 0; l < ORDER; ++l) {
    bad |= (uint32_t)v[l] >= (uint32_t)k.dim[l];          // extents are below 2^31: a negative coordinate is beyond them too
    key |= ((uint64_t)(uint32_t)v[l] & ((1ull << k.bits[l]) - 1)) << k.shift[l];
  }
  return key;
}

// Exclusive scan of one value per thread over the CTA (any number of whole warps); s_warp holds 32 words.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *s_warp, uint32_t *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  uint32_t inc = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, inc, off);
    if (lane >= off) inc += t;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < warps ? s_warp[lane] : 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += t;
    }
    if (lane < warps) s_warp[lane] = w;        // inclusive over warps
  }
  __syncthreads();
  const uint32_t before = warp > 0 ? s_warp[warp - 1] : 0;
  if (total) *total = s_warp[warps - 1];
  __syncthreads();
  return before + inc - v;
}

struct LevelPlan {
  int order;
  int attr[COMET_MAX_ORDER];
  int shift[COMET_MAX_ORDER];
  int bits[COMET_MAX_ORDER];
  int counted[COMET_MAX_ORDER];     // index of the level's node counter (-1: positions are entry ranks or dense)
  int ncounted;
};

__device__ __forceinline__ bool is_head(uint64_t k, uint64_t kprev, bool first, int shift) {
  return first || (k >> shift) != (kprev >> shift);
}

// Entries per tile of the level counts: level_count_kernel and level_emit_kernel (pack.cu) and the one launch of
// pack_small.cu count and place nodes in the same tiles.
constexpr int kLevelThreads = 256;
constexpr int kLevelItems = 8;
constexpr int kLevelTile = kLevelThreads * kLevelItems;

struct LevelOut {
  int32_t *pos[COMET_MAX_ORDER];
  int32_t *crd[COMET_MAX_ORDER];
  void *val;                   // fp64 or fp32, as the COO values
  int64_t dim0;                // extent of level 0 (for a dense root)
  uint32_t nodes[COMET_MAX_ORDER];   // node count of every counted level (indexed by level)
};

// Small inputs (pack_small.cu): keys, sort and level counts in one cooperative launch. `tmp` holds pack_small_bytes();
// the call waits for the stream, after which the handle's pinned words hold what pack.cu reads from them (0 range error, 1
// duplicate, 8 + l nodes of level l) and `out` the sorted entries and the scanned counts per tile of kLevelTile entries.
// COMET_ERR_UNSUPPORTED_FORMAT: the driver refused the launch, as it does where the context has fewer SMs than the device
// (nothing was written; COMET_PACK_SMALL=0 stands for such a refusal): take the general path.
struct PackSmallSorted {
  uint64_t *keys;
  uint32_t *pay;
  uint32_t *counts;
};
bool pack_small_applies(Context *ctx, int order, int total_bits, int64_t n);
size_t pack_small_bytes(int order, int64_t n);
comet_status_t pack_small_sort(Context *ctx, int order, const CoordPtrs &c, const KeyLayout &k, const LevelPlan &plan,
                               const uint32_t *val32, int64_t n, char *tmp, PackSmallSorted *out, cudaStream_t s);

// Larger inputs of distinct keys (pack_split.cu): split by sampled keys, sorted in shared memory. `tmp` holds
// pack_split_bytes(); nothing waits. direct null: `sorted` receives the sorted keys and values (inside `tmp`); otherwise the
// tensor's arrays, which are written (CSR [D,CU] and sorted coordinates [CN,S..]: no level needs a count). The status words
// tell afterwards: with kStatusOverflow the input did not fit this path and what was written is void.
struct PackSplitSorted {
  uint64_t *keys;
  void *val;
};
bool pack_split_applies(int order, int total_bits, int64_t n);
size_t pack_split_bytes(int64_t n);
comet_status_t pack_split_sort(Context *ctx, int order, const CoordPtrs &c, const KeyLayout &k, const LevelPlan &plan, const void *val,
                               int dtype, int64_t n, char *tmp, const LevelOut *direct, PackSplitSorted *sorted, cudaStream_t s);

}  // namespace comet

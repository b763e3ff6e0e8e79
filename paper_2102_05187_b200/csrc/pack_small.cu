// comet_pack for small inputs: keys, sort and level counts in ONE launch.
//
// A packing of some ten thousand entries spends its time on launches, not on data: the general path (pack.cu) takes five
// launches per 8-bit digit, each of them 2 to 7 us of latency for kilobytes of work. Here a cooperative grid of at most one
// CTA per SM keeps a tile of the entries per CTA and goes through the same steps with grid-wide barriers in between:
// per digit count and rank the tile, publish its 256 counts, barrier, add up the counts of the tiles (every CTA for
// itself: a few hundred words per digit), scatter, barrier. Then the level counts of pack.cu's 2,048-entry tiles, scanned,
// so that its emit kernel can follow. The node counts and the error flags go straight to the handle's pinned host words.
// What bounds it is the latency of the steps (about 9 us per digit: two grid barriers, two rounds through L2, the ranking).
// Measured against the general path, whole comet_pack calls: 500 entries, order 3 162 -> 52 us; 60,000 entries of order 3
// (four digits) packed and contracted once 325 -> 112 us; 0.42 M entries, five digits 323 -> 135 us. Beyond 8 entries per
// thread pack_split.cu is faster (620,000 entries 142 us here with 16, 106 there).
//
// The barriers are cooperative groups' (the launch guarantees that all CTAs are resident); nothing else waits.
#include <cooperative_groups.h>

#include <stdlib.h>

#include "common.cuh"
#include "kernels.cuh"
#include "pack_common.cuh"

namespace comet {

namespace cg = cooperative_groups;

constexpr int kSmallThreads = 512;
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kSmallMaxItems = 8;
constexpr int64_t kSmallMax = (int64_t)kSmCount * kSmallThreads * kSmallMaxItems;     // 0.6 M entries

template <int ORDER> struct SmallArgs {
  CoordPtrs c;
  KeyLayout k;
  LevelPlan plan;
  const uint32_t *val32;             // 32-bit values, or null: the payload is the entry's index
  uint32_t n, tiles;
  uint64_t *keys[2];
  uint32_t *pay[2];
  uint32_t *table;                   // tiles x 256
  uint32_t *counts;                  // ORDER x level_tiles: node counts, then their exclusive scan
  uint32_t level_tiles;
  int32_t *host;                     // pinned host words: 0 range error, 1 duplicate, 8 + l nodes of level l
};

template <int ORDER, int ITEMS>
__global__ void __launch_bounds__(kSmallThreads, 1) pack_small_kernel(const SmallArgs<ORDER> a) {
  cg::grid_group grid = cg::this_grid();
  __shared__ uint32_t s_cnt[kSmallWarps][256];
  __shared__ uint32_t s_half[2][2][256];          // [half][total, before]
  __shared__ uint32_t s_off[256];
  __shared__ uint32_t s_warp[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t tile = blockIdx.x;
  const uint32_t tile_base = tile * (kSmallThreads * ITEMS), warp_base = tile_base + warp * (32 * ITEMS);
  const uint32_t pads = tile_base + kSmallThreads * ITEMS > a.n ? tile_base + kSmallThreads * ITEMS - a.n : 0;
  const unsigned lt = (1u << lane) - 1u;
  int cur = 0;
  for (int shift = 0; shift < a.k.total_bits; shift += 8) {
    uint64_t key[ITEMS];
    uint32_t pay[ITEMS], rank[ITEMS];
    if (shift == 0) {
      bool bad = false;
#pragma unroll
      for (int r = 0; r < ITEMS; ++r) {
        const uint32_t i = warp_base + r * 32 + lane, j = i < a.n ? i : a.n - 1;
        key[r] = entry_key<ORDER>(a.c, a.k, j, bad);
        pay[r] = a.val32 ? __ldcs(a.val32 + j) : j;
      }
      if (bad) *reinterpret_cast<volatile int32_t *>(a.host) = 1;
    } else {
      const uint64_t *kin = a.keys[cur];
      const uint32_t *pin = a.pay[cur];
#pragma unroll
      for (int r = 0; r < ITEMS; ++r) {           // written by other SMs in this launch: read past L1
        const uint32_t i = warp_base + r * 32 + lane, j = i < a.n ? i : a.n - 1;
        key[r] = __ldcg(kin + j);
        pay[r] = __ldcg(pin + j);
      }
    }
    for (int x = tid; x < kSmallWarps * 256; x += kSmallThreads) (&s_cnt[0][0])[x] = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {             // slots past the end rank behind every entry of the tile, in digit 255
      const bool in = warp_base + r * 32 + lane < a.n;
      const uint32_t d = in ? (uint32_t)(key[r] >> shift) & 255u : 255u;
      const unsigned peers = __match_any_sync(0xffffffffu, d);
      const int leader = __ffs(peers) - 1;
      uint32_t old = 0;
      if (lane == leader) old = atomicAdd(&s_cnt[warp][d], (uint32_t)__popc(peers));
      old = __shfl_sync(0xffffffffu, old, leader);
      rank[r] = old + __popc(peers & lt);
      __syncwarp();
    }
    __syncthreads();
    if (tid < 256) {
      uint32_t run = 0;
#pragma unroll
      for (int w = 0; w < kSmallWarps; ++w) {
        const uint32_t c = s_cnt[w][tid];
        s_cnt[w][tid] = run;
        run += c;
      }
      __stcg(a.table + tile * 256 + tid, run - (tid == 255 ? pads : 0u));
    }
    grid.sync();
    {
      // digit `tid & 255`: entries of it in all tiles and in the tiles in front, half of the tiles per thread
      const int d = tid & 255, h = tid >> 8;
      uint32_t total = 0, before = 0;
      uint32_t t = h;
      for (; t + 14 < a.tiles; t += 16) {
        uint32_t v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldcg(a.table + (t + 2 * u) * 256 + d);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          total += v[u];
          if (t + 2 * u < tile) before += v[u];
        }
      }
      for (; t < a.tiles; t += 2) {
        const uint32_t v = __ldcg(a.table + t * 256 + d);
        total += v;
        if (t < tile) before += v;
      }
      s_half[h][0][d] = total;
      s_half[h][1][d] = before;
    }
    __syncthreads();
    const uint32_t all = tid < 256 ? s_half[0][0][tid] + s_half[1][0][tid] : 0;
    const uint32_t start = block_exclusive_scan(all, s_warp, nullptr);
    if (tid < 256) s_off[tid] = start + s_half[0][1][tid] + s_half[1][1][tid];
    __syncthreads();
    uint64_t *kout = a.keys[cur ^ 1];
    uint32_t *pout = a.pay[cur ^ 1];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      if (warp_base + r * 32 + lane < a.n) {
        const uint32_t d = (uint32_t)(key[r] >> shift) & 255u;
        const uint32_t at = s_off[d] + s_cnt[warp][d] + rank[r];
        __stcg(kout + at, key[r]);
        __stcg(pout + at, pay[r]);
      }
    }
    cur ^= 1;
    grid.sync();
  }

  // node counts per tile of pack.cu's emit kernel, duplicates
  const uint64_t *keys = a.keys[cur];
  bool dup = false;
  for (uint32_t lv = blockIdx.x; lv < a.level_tiles; lv += gridDim.x) {
    uint32_t mine[ORDER];
#pragma unroll
    for (int l = 0; l < ORDER; ++l) mine[l] = 0;
    constexpr int kRounds = kLevelTile / kSmallThreads;
    static_assert(kRounds * kSmallThreads == kLevelTile, "whole rounds of the CTA per level tile");
    uint64_t k[kRounds], kp[kRounds];
#pragma unroll
    for (int u = 0; u < kRounds; ++u) {
      const uint32_t p = lv * kLevelTile + u * kSmallThreads + tid, q = p < a.n ? p : a.n - 1;
      k[u] = __ldcg(keys + q);
      kp[u] = __ldcg(keys + (q > 0 ? q - 1 : 0));
    }
#pragma unroll
    for (int u = 0; u < kRounds; ++u) {
      const uint32_t p = lv * kLevelTile + u * kSmallThreads + tid;
      if (p < a.n) {
        dup |= (p > 0) & (k[u] == kp[u]);
#pragma unroll
        for (int l = 0; l < ORDER; ++l)
          if (a.plan.counted[l] >= 0 && is_head(k[u], kp[u], p == 0, a.plan.shift[l])) mine[l] += 1;
      }
    }
#pragma unroll
    for (int l = 0; l < ORDER; ++l) {
      if (a.plan.counted[l] < 0) continue;
      uint32_t total;
      block_exclusive_scan(mine[l], s_warp, &total);
      if (tid == 0) __stcg(a.counts + l * a.level_tiles + lv, total);
    }
  }
  if (dup) reinterpret_cast<volatile int32_t *>(a.host)[1] = 1;
  if (a.plan.ncounted == 0) return;
  grid.sync();
  for (int l = blockIdx.x; l < ORDER; l += gridDim.x) {
    int counted = -1;
#pragma unroll
    for (int x = 0; x < ORDER; ++x) if (x == l) counted = a.plan.counted[x];
    if (counted < 0) continue;
    uint32_t carry = 0;
    for (uint32_t base = 0; base < a.level_tiles; base += kSmallThreads) {
      const uint32_t i = base + tid;
      const uint32_t v = i < a.level_tiles ? __ldcg(a.counts + l * a.level_tiles + i) : 0;
      uint32_t total;
      const uint32_t ex = block_exclusive_scan(v, s_warp, &total);
      if (i < a.level_tiles) a.counts[l * a.level_tiles + i] = carry + ex;
      carry += total;
    }
    if (tid == 0) reinterpret_cast<volatile int32_t *>(a.host)[8 + l] = (int32_t)carry;
  }
}

static int small_items(int64_t n) {
  const int64_t per = ceil_div(n, (int64_t)kSmCount * kSmallThreads);
  return per <= 2 ? 2 : per <= 4 ? 4 : 8;
}

bool pack_small_applies(Context *ctx, int order, int total_bits, int64_t n) {
  if (n < 1 || n > kSmallMax || total_bits < 1 || order < 2) return false;
  // the launch needs an SM per tile; a device (or a slice of one) with fewer takes the general path
  if (ctx->sm_count == 0) {
    int sms = 0, coop = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device) != cudaSuccess) { cudaGetLastError(); sms = -1; }
    ctx->sm_count = coop && sms > 0 ? sms : -1;
  }
  return ceil_div(n, (int64_t)kSmallThreads * small_items(n)) <= ctx->sm_count;
}

// keys_a/b and pay_a/b, the digit table and the level counts
size_t pack_small_bytes(int order, int64_t n) {
  return 2 * align_up((size_t)n * 8, 256) + 2 * align_up((size_t)n * 4, 256) + (size_t)kSmCount * 256 * 4 +
         align_up((size_t)order * ceil_div(n, kLevelTile) * 4, 256);
}

template <int ORDER>
static cudaError_t launch_small(SmallArgs<ORDER> a, int items, cudaStream_t s) {
  a.tiles = (uint32_t)ceil_div((int64_t)a.n, (int64_t)kSmallThreads * items);
  void *args[] = {&a};
  const void *kernel = items == 2 ? (const void *)pack_small_kernel<ORDER, 2> : items == 4 ? (const void *)pack_small_kernel<ORDER, 4>
                                         : (const void *)pack_small_kernel<ORDER, 8>;
  return cudaLaunchCooperativeKernel(kernel, dim3(a.tiles), dim3(kSmallThreads), args, 0, s);
}

template <int ORDER>
static cudaError_t run_small(const CoordPtrs &c, const KeyLayout &k, const LevelPlan &plan, const uint32_t *val32, int64_t n, char *tmp,
                             int32_t *host, PackSmallSorted *out, cudaStream_t s) {
  SmallArgs<ORDER> a{};
  a.c = c; a.k = k; a.plan = plan; a.val32 = val32; a.n = (uint32_t)n; a.host = host;
  auto take = [&](size_t bytes) { char *p = tmp; tmp += align_up(bytes, 256); return p; };
  for (int x = 0; x < 2; ++x) a.keys[x] = (uint64_t *)take((size_t)n * 8);
  for (int x = 0; x < 2; ++x) a.pay[x] = (uint32_t *)take((size_t)n * 4);
  a.table = (uint32_t *)take((size_t)kSmCount * 256 * 4);
  a.counts = (uint32_t *)tmp;
  a.level_tiles = (uint32_t)ceil_div(n, kLevelTile);
  const int at = ((k.total_bits + 7) / 8) & 1;     // the buffer that the last digit's scatter writes
  out->keys = a.keys[at];
  out->pay = a.pay[at];
  out->counts = a.counts;
  host[0] = host[1] = 0;
  return launch_small<ORDER>(a, small_items(n), s);
}

comet_status_t pack_small_sort(Context *ctx, int order, const CoordPtrs &c, const KeyLayout &k, const LevelPlan &plan,
                               const uint32_t *val32, int64_t n, char *tmp, PackSmallSorted *out, cudaStream_t s) {
  const char *allowed = getenv("COMET_PACK_SMALL");
  cudaError_t e;
  if (allowed && allowed[0] == '0') e = cudaErrorCooperativeLaunchTooLarge;
  else if (order == 2) e = run_small<2>(c, k, plan, val32, n, tmp, ctx->h_pinned, out, s);
  else if (order == 3) e = run_small<3>(c, k, plan, val32, n, tmp, ctx->h_pinned, out, s);
  else e = run_small<4>(c, k, plan, val32, n, tmp, ctx->h_pinned, out, s);
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
    cudaGetLastError();
    return COMET_ERR_UNSUPPORTED_FORMAT;
  }
  if (e != cudaSuccess) return cuda_fail(ctx, e);
  ctx->launches += 1;
  COMET_CUDA_TRY(ctx, cudaStreamSynchronize(s));
  return COMET_OK;
}

}  // namespace comet

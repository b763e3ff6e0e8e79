// comet_pack of larger inputs: the entries are split by sampled keys, twice, and the pieces sorted in shared memory.
//
// The keys of a packing are distinct (equal ones are an error), so nothing has to be stable and an entry moves three
// times whatever the number of key bits, where the radix sort of pack.cu moves it once per 8 bits and gathers 64-bit
// values at the end. Splitters are sampled, not digits, so that power-law modes make no large pieces:
//   1. a sample of the keys, 32 per coarse bucket (32 to 512 buckets), is put in order;
//   2. every tile of 4,096 entries forms its keys, finds each one's bucket in a search tree of the splitters, counts,
//      takes room in every bucket with one atomic add, and writes its runs as records of key and value (16 bytes);
//   3. a CTA per coarse bucket samples and sorts again: splitters of fine buckets of about 1,400 entries;
//   4. the same split inside every coarse bucket, into regions of 3,584 records per fine bucket;
//   5. a CTA per fine bucket: the 32 samples of the bucket and linear interpolation between them give each entry one
//      of 2,048 cells in key order (64 between two samples, less than one entry each on average), and a count of the
//      smaller keys of its cell gives its place.
// Formats whose levels all have an entry per node (CSR, sorted coordinates) are written by step 5 itself; the others
// get sorted keys and values, for the level kernels of pack.cu.
//
// A bucket that its region cannot hold (2.5 times the expected size) raises a flag, nothing is written beyond a region, and
// pack.cu sorts again. How often, from the distribution of the samples' spacings (Beta) summed over the buckets: at most
// one packing of distinct keys in 50,000 up to 40 M entries, 2 in 10,000 up to 90 M, 1 in 1,000 at 100 M and 9 in 1,000 at the
// limit of 114.7 M, where a coarse bucket has up to 256 fine ones and still 4,096 samples. Which entries are sampled depends on their
// number alone, so that an input whose order misleads the samples does so on every call. No CTA waits for another.
//
// The splits are bound by the steps that their barriers keep apart (search 40 us, counting 15 to 25, copies out 20 to 40,
// reading and ordering the records 80, of 160; L1 59 %, issue 42 to 52 %, most stalls at barriers), the last step by the same, the
// load/store pipe (71 %) and instruction issue (53 %). Measured against the radix sort, whole comet_pack calls: 19.8 M entries to CSR, fp64 1431 ->
// 726 us, fp32 1215 -> 712; 100 M to sorted coordinates 9157 -> 4020; 50 M to CSF 3957 -> 2360; 3 M to CSF 423 -> 250.
// Tiles of 2,048 records, three to five CTAs per SM and a CTA per tile all gave 160 to 190 us for a split.
#include "common.cuh"
#include "kernels.cuh"
#include "pack_common.cuh"

#include <stddef.h>
#include <stdlib.h>

namespace comet {

constexpr int kSplitThreads = 512;
constexpr int kSplitItems = 8;
constexpr int kSplitTile = kSplitThreads * kSplitItems;
constexpr int kSplitMaxBuckets = 512;
constexpr int kSplitOver = 32;                   // samples per bucket
constexpr int kSplitMean = 1400;                 // entries per fine bucket
constexpr int kSplitCap = 3584;                  // records of a fine bucket's region
constexpr int kSplitCursorStride = 32;           // words between the cursors of coarse buckets: a 128-byte line each
constexpr int kSplitBulkLevels = 8;              // up to 256 buckets a run leaves as one bulk copy
constexpr int kSampleThreads = 1024;
constexpr int kPieceCells = 64;                  // cells between two samples
constexpr int kSplitCells = 32 * kPieceCells;

struct __align__(16) SplitRecord {
  uint64_t key, val;                             // val: a double's or (low half) a float's bits
};

struct SplitShape {
  int64_t n;
  int total_bits;                                // of a key
  int k1, k2;                                    // log2 of the coarse buckets, of the most fine buckets per coarse one
  int64_t cap1;                                  // records of a coarse bucket's region
  int64_t fine_max, tile_max;                    // bounds of the numbers of fine buckets and of tiles in step 4
};

struct SplitBuffers {
  uint32_t *cursor1, *cursor2;                   // entries placed so far, per bucket
  uint64_t *drawn;                               // samples of all entries as drawn
  uint64_t *samples1, *samples2;                 // samples in order: of all entries, of every coarse bucket
  uint32_t *coarse_start, *fine_base;            // first entry, first fine bucket of every coarse bucket
  uint4 *tile_map;                               // step 4: a tile's coarse bucket and fine buckets, first entry, entries, first fine bucket
  uint32_t *fine_map;                            // coarse bucket of a fine bucket
  uint32_t *totals;                              // tiles of step 4, fine buckets
  uint4 *edges;                                  // CSR: first row, last row, first position, entries of a fine bucket
  SplitRecord *rec1, *rec2;
  int32_t *status;
};

static SplitShape split_shape(int64_t n, int total_bits) {
  SplitShape s{};
  s.n = n;
  s.total_bits = total_bits;
  const int64_t want = ceil_div(n, kSplitMean);
  s.k1 = 5;
  while (s.k1 < 9 && ceil_div(want, 1ll << s.k1) > 128) ++s.k1;
  const int64_t mean2 = ceil_div(want, 1ll << s.k1);
  s.k2 = 5;                                      // a bucket a lane at least
  while (s.k2 < 8 && (1ll << s.k2) < mean2 * 27 / 20 + 2) ++s.k2;
  s.cap1 = align_up((size_t)(n / (1ll << s.k1) * 5 / 2 + kSplitTile), 16);
  s.fine_max = n / kSplitMean + (1ll << s.k1);
  s.tile_max = n / kSplitTile + (1ll << s.k1);
  return s;
}

// Spreads sample numbers over 32 bits: lowbias32 of C. Wellons' "Hash Prospector", shifts and multipliers as published.
__device__ __forceinline__ uint32_t sample_hash(uint32_t x) {
  x ^= x >> 16; x *= 0x7feb352du;
  x ^= x >> 15; x *= 0x846ca68bu;
  return x ^ (x >> 16);
}

// Sorts kSampleThreads * PER keys in shared memory (bitonic). A thread holds PER consecutive keys in registers: steps
// between keys of one thread need nothing, between lanes shuffles, and only wider ones shared memory and barriers
// (4,096 keys: 46 us with every step through shared memory).
template <int PER>
__device__ __forceinline__ void sort_samples(uint64_t *k) {
  const int tid = threadIdx.x;
  uint64_t v[PER];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < PER; ++r) v[r] = k[tid * PER + r];
  for (int size = 2; size <= kSampleThreads * PER; size <<= 1) {
    int half = size >> 1;
    if (half >= 32 * PER) {
      __syncthreads();
#pragma unroll
      for (int r = 0; r < PER; ++r) k[r * kSampleThreads + tid] = v[r];       // key tid * PER + r, without bank conflicts
      for (; half >= 32 * PER; half >>= 1) {
        const int far = tid ^ (half / PER);      // the thread that holds the other keys
        const bool up = ((tid * PER) & size) == 0, low = tid < far;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < PER; ++r) {
          const uint64_t o = k[r * kSampleThreads + far];
          if ((o < v[r]) == (up == low)) v[r] = o;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < PER; ++r) k[r * kSampleThreads + tid] = v[r];
      }
    }
    for (; half >= PER; half >>= 1) {
      const int far = half / PER;
      const bool up = ((tid * PER) & size) == 0, low = (tid & far) == 0;
#pragma unroll
      for (int r = 0; r < PER; ++r) {
        const uint64_t o = __shfl_xor_sync(0xffffffffu, (unsigned long long)v[r], far);
        if ((o < v[r]) == (up == low)) v[r] = o;
      }
    }
#pragma unroll
    for (int h = PER >> 1; h > 0; h >>= 1) {
      if (h > half) continue;
#pragma unroll
      for (int r = 0; r < PER; ++r)
        if ((r & h) == 0) {
          const bool up = ((tid * PER + r) & size) == 0;
          const uint64_t x = v[r], y = v[r + h];
          if ((x > y) == up) { v[r] = y; v[r + h] = x; }
        }
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < PER; ++r) k[tid * PER + r] = v[r];
  __syncthreads();
}

// Keys that sort_samples sorts for `count` of them (1, 2 or 4 a thread), and the sort.
constexpr int kMostSamples = 4 * kSampleThreads;
__device__ __forceinline__ int sample_room(int count) { return count <= kSampleThreads ? kSampleThreads : count <= 2 * kSampleThreads ? 2 * kSampleThreads : kMostSamples; }
__device__ __forceinline__ void sort_samples(uint64_t *k, int room) {
  if (room == kSampleThreads) sort_samples<1>(k);
  else if (room == 2 * kSampleThreads) sort_samples<2>(k);
  else sort_samples<4>(k);
}

// Which of 2^levels - 1 splitters, counted from 1, stands at node i >= 1 of their search tree (children: 2i, 2i + 1).
__device__ __forceinline__ int heap_rank(int i, int levels) {
  const int depth = 31 - __clz(i), q = i - (1 << depth);
  return (2 * q + 1) << (levels - 1 - depth);
}

// ---------------------------------------------------------------------------------------------- samples
// The samples of step 1, and after them in order. One CTA that sorts them would be the only one at work (25 us for 4,096);
// here a warp counts the smaller ones of a key, all of them in shared memory of every CTA.
template <int ORDER>
__global__ void __launch_bounds__(kSplitThreads) split_sample_coarse_kernel(CoordPtrs c, KeyLayout k, SplitShape sh, SplitBuffers b) {
  const int f1 = 1 << sh.k1, i = blockIdx.x * kSplitThreads + threadIdx.x;
  bool ignored = false;
  if (i < f1) b.cursor1[i * kSplitCursorStride] = 0;
  if (i < f1 * kSplitOver)
    b.drawn[i] = entry_key<ORDER>(c, k, (int64_t)(((uint64_t)sample_hash(i) * (uint64_t)sh.n) >> 32), ignored);
}
__global__ void __launch_bounds__(kSampleThreads) split_rank_samples_kernel(SplitShape sh, SplitBuffers b) {
  extern __shared__ __align__(16) uint64_t s_keys[];
  const int count = kSplitOver << sh.k1, tid = threadIdx.x, lane = tid & 31;
  for (int i = 2 * tid; i < count; i += 2 * kSampleThreads)
    *reinterpret_cast<ulonglong2 *>(s_keys + i) = *reinterpret_cast<const ulonglong2 *>(b.drawn + i);
  __syncthreads();
  for (int i = (blockIdx.x * kSampleThreads + tid) >> 5; i < count; i += gridDim.x * (kSampleThreads / 32)) {
    const uint64_t key = s_keys[i];
    int rank = 0;
    int j = lane;
#pragma unroll 8
    for (; j < (i & ~31); j += 32) rank += s_keys[j] <= key ? 1 : 0;          // equal keys keep their order
    { const uint64_t o = s_keys[j]; rank += (o < key || (o == key && j < i)) ? 1 : 0; }
#pragma unroll 8
    for (j += 32; j < count; j += 32) rank += s_keys[j] < key ? 1 : 0;
    rank = __reduce_add_sync(0xffffffffu, rank);
    if (lane == 0) b.samples1[rank] = key;
  }
}
// Where coarse bucket i's keys begin (i up to the number of buckets).
__device__ __forceinline__ uint64_t coarse_bound(const SplitShape &sh, const SplitBuffers &b, int i) {
  return i == 0 ? 0 : i >= 1 << sh.k1 ? 1ull << sh.total_bits : b.samples1[i * kSplitOver];
}

__device__ __forceinline__ uint32_t coarse_count(const SplitShape &sh, const SplitBuffers &b, int c) {
  const uint32_t got = b.cursor1[c * kSplitCursorStride];
  return got < (uint32_t)sh.cap1 ? got : (uint32_t)sh.cap1;
}
__device__ __forceinline__ uint32_t fine_count(const SplitShape &sh, uint32_t entries) {
  const uint32_t want = (entries + kSplitMean - 1) / kSplitMean, most = 1u << sh.k2;
  return want < most ? want : most;
}

__global__ void __launch_bounds__(kSampleThreads, 2) split_sample_fine_kernel(SplitShape sh, SplitBuffers b) {
  extern __shared__ __align__(16) uint64_t s_keys[];
  const int f1 = 1 << sh.k1, most = 1 << sh.k2;
  if ((int)blockIdx.x == f1) {                   // one more CTA: where the coarse buckets start, and step 4's tiles
    __shared__ uint32_t s_warp[32];
    const int c = threadIdx.x;
    const uint32_t m = c < f1 ? coarse_count(sh, b, c) : 0;
    const uint32_t fine = fine_count(sh, m), tiles = (m + kSplitTile - 1) / kSplitTile;
    uint32_t fines, all_tiles;
    const uint32_t start = block_exclusive_scan(m, s_warp, nullptr);
    const uint32_t base = block_exclusive_scan(fine, s_warp, &fines);
    const uint32_t tile0 = block_exclusive_scan(tiles, s_warp, &all_tiles);
    if (c <= f1) { b.coarse_start[c] = start; b.fine_base[c] = base; }
    for (uint32_t t = 0; t < tiles; ++t) b.tile_map[tile0 + t] = make_uint4(c | fine << 16, t * kSplitTile, m - t * kSplitTile < kSplitTile ? m - t * kSplitTile : kSplitTile, base);
    for (uint32_t t = 0; t < fine; ++t) b.fine_map[base + t] = c;
    if (threadIdx.x == 0) {
      // no tile for step 4 where step 2's regions have holes in which no record lies, or hold records whose keys are no keys
      b.totals[0] = b.status[kStatusOverflow] | b.status[kStatusRange] ? 0 : all_tiles;
      b.totals[1] = fines;
    }
    return;
  }
  const int c = blockIdx.x;
  for (int i = threadIdx.x; i < most; i += kSampleThreads) b.cursor2[((size_t)c << sh.k2) + i] = 0;
  const uint32_t m = coarse_count(sh, b, c);
  const int fine = fine_count(sh, m), count = fine * kSplitOver;
  if (!fine) return;
  // A coarse bucket much larger than the mean makes do with the samples that are sorted quickly (with up to 8,192 the few
  // that needed them took 47 us, the others 30): some then stand twice among its `count`.
  const int drawn = count < kMostSamples ? count : kMostSamples;
  const int room = sample_room(drawn);
  const SplitRecord *rec = b.rec1 + (size_t)c * sh.cap1;
  for (int i = threadIdx.x; i < room; i += kSampleThreads)
    s_keys[i] = i < drawn ? rec[((uint64_t)sample_hash(i + 0x10000u * (c + 1)) * m) >> 32].key : ~0ull;
  sort_samples(s_keys, room);
  uint64_t *samples = b.samples2 + ((size_t)c << sh.k2) * kSplitOver;
  for (int i = threadIdx.x; i < count; i += kSampleThreads) samples[i] = s_keys[(int64_t)i * drawn / count];
}

// ---------------------------------------------------------------------------------------------- splits
struct SplitJob {                                // a tile: entries [first, first + valid) of coarse bucket `bucket`
  int64_t first;
  int valid;
  int bucket;                                    // (step 2: 0)
  int live;                                      // buckets it is split into
  int64_t region0;                               // where the first of these has its region
};

// What a tile is read from. `load` asks for the entries of a tile, `keys` forms their keys, `value` reads the value of the
// thread's entry t, which is t * kSplitThreads + threadIdx.x unless the tile is full, where the order does not matter.
template <int ORDER>
struct SplitCoo {                                // step 2: the caller's arrays
  CoordPtrs c;
  KeyLayout k;
  const void *val;
  bool f32, wide;                                // wide: every coordinate array is aligned to 16 bytes
  struct Raw { int32_t c[ORDER][kSplitItems]; };

  static __device__ __forceinline__ int64_t tiles(const SplitShape &sh, const SplitBuffers &) { return (sh.n + kSplitTile - 1) / kSplitTile; }
  __device__ __forceinline__ SplitJob job(const SplitShape &sh, const SplitBuffers &, int64_t tile) const {
    const int64_t first = tile * kSplitTile;
    return SplitJob{first, sh.n - first < kSplitTile ? (int)(sh.n - first) : kSplitTile, 0, 1 << sh.k1, 0};
  }
  static __device__ __forceinline__ const uint64_t *samples(const SplitShape &, const SplitBuffers &b, int) { return b.samples1; }
  static __device__ __forceinline__ uint32_t *cursor(const SplitShape &, const SplitBuffers &b, int, int d) { return b.cursor1 + d * kSplitCursorStride; }

  __device__ __forceinline__ void load(const SplitShape &, const SplitBuffers &, const SplitJob &j, Raw &raw) const {
    const int tid = threadIdx.x;
    if (wide && j.valid == kSplitTile) {         // four entries in a row per access (a tile starts at a multiple of four)
      static_assert(kSplitItems % 4 == 0 && kSplitTile % 4 == 0, "");
#pragma unroll
      for (int l = 0; l < ORDER; ++l)
#pragma unroll
        for (int g = 0; g < kSplitItems / 4; ++g) {
          const int4 v = __ldcs(reinterpret_cast<const int4 *>(c.p[l] + j.first) + g * kSplitThreads + tid);
          raw.c[l][4 * g] = v.x; raw.c[l][4 * g + 1] = v.y; raw.c[l][4 * g + 2] = v.z; raw.c[l][4 * g + 3] = v.w;
        }
      return;
    }
#pragma unroll
    for (int t = 0; t < kSplitItems; ++t) {
      const int i = t * kSplitThreads + tid;
      const int64_t at = j.first + (i < j.valid ? i : j.valid - 1);
#pragma unroll
      for (int l = 0; l < ORDER; ++l) raw.c[l][t] = __ldcs(c.p[l] + at);
    }
  }
  __device__ __forceinline__ void keys(const Raw &raw, uint64_t (&key)[kSplitItems], int32_t *status) const {
    bool bad = false;
#pragma unroll
    for (int t = 0; t < kSplitItems; ++t) key[t] = 0;
#pragma unroll
    for (int l = 0; l < ORDER; ++l) {
      const uint32_t dim = (uint32_t)k.dim[l];
#pragma unroll
      for (int t = 0; t < kSplitItems; ++t) {
        bad |= (uint32_t)raw.c[l][t] >= dim;     // such a key is no key; nothing is made of it
        key[t] |= (uint64_t)(uint32_t)raw.c[l][t] << k.shift[l];
      }
    }
    if (bad) atomicOr(status + kStatusRange, 1);
  }
  __device__ __forceinline__ uint64_t value(const Raw &, const SplitJob &j, int t) const {
    const int64_t i = j.first + (wide && j.valid == kSplitTile ? ((t >> 2) * kSplitThreads + threadIdx.x) * 4 + (t & 3) : t * kSplitThreads + threadIdx.x);
    return f32 ? (uint64_t)__ldcs(static_cast<const uint32_t *>(val) + i) : (uint64_t)__ldcs(static_cast<const unsigned long long *>(val) + i);
  }
};

struct SplitRec {                                // step 4: the coarse buckets' regions
  struct Raw { SplitRecord r[kSplitItems]; };

  static __device__ __forceinline__ int64_t tiles(const SplitShape &, const SplitBuffers &b) { return b.totals[0]; }
  __device__ __forceinline__ SplitJob job(const SplitShape &sh, const SplitBuffers &b, int64_t tile) const {
    const uint4 m = b.tile_map[tile];
    return SplitJob{m.y, (int)m.z, (int)(m.x & 0xffffu), (int)(m.x >> 16), (int64_t)m.w * kSplitCap};
  }
  static __device__ __forceinline__ const uint64_t *samples(const SplitShape &sh, const SplitBuffers &b, int c) {
    return b.samples2 + ((size_t)c << sh.k2) * kSplitOver;
  }
  static __device__ __forceinline__ uint32_t *cursor(const SplitShape &sh, const SplitBuffers &b, int c, int d) {
    return b.cursor2 + ((size_t)c << sh.k2) + d;
  }
  __device__ __forceinline__ void load(const SplitShape &sh, const SplitBuffers &b, const SplitJob &j, Raw &raw) const {
    const SplitRecord *rec = b.rec1 + (size_t)j.bucket * sh.cap1 + j.first;
#pragma unroll
    for (int t = 0; t < kSplitItems; ++t) {
      const int i = t * kSplitThreads + threadIdx.x;
      const ulonglong2 two = __ldcs(reinterpret_cast<const ulonglong2 *>(rec + (i < j.valid ? i : j.valid - 1)));
      raw.r[t] = SplitRecord{two.x, two.y};
    }
  }
  __device__ __forceinline__ void keys(const Raw &raw, uint64_t (&key)[kSplitItems], int32_t *) const {
#pragma unroll
    for (int t = 0; t < kSplitItems; ++t) key[t] = raw.r[t].key;
  }
  __device__ __forceinline__ uint64_t value(const Raw &raw, const SplitJob &, int t) const { return raw.r[t].val; }
};

struct SplitShared {
  SplitRecord rec[kSplitTile];                   // the tile, bucket by bucket
  uint64_t heap[kSplitMaxBuckets];
  uint32_t count[kSplitMaxBuckets];
  uint32_t start[kSplitMaxBuckets];
  // only where runs are written by the threads:
  int64_t delta[kSplitMaxBuckets];               // record index of a bucket's run minus its start in the tile; < 0: no room
  uint16_t bucket[kSplitTile];
};

// Steps 2 and 4. A CTA goes through a row of tiles and asks for the next one before it writes the last (with a CTA per
// tile it waited for its maps, its splitters and its entries in turn: 4,096 records per 5 us and SM whatever the occupancy).
template <class Src>
__global__ void __launch_bounds__(kSplitThreads, 2) split_kernel(Src src, SplitShape sh, SplitBuffers b, int levels, uint32_t cap,
                                                                 SplitRecord *__restrict__ out) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  SplitShared &s = *reinterpret_cast<SplitShared *>(s_raw);
  const int tid = threadIdx.x, lane = tid & 31, buckets = 1 << levels;
  const int64_t tiles = Src::tiles(sh, b);
  int64_t tile = tiles * blockIdx.x / gridDim.x;
  const int64_t end = tiles * (blockIdx.x + 1) / gridDim.x;
  if (tile >= end) return;
  // Runs of 16 records and more on average leave as one bulk copy each: the records pass the load/store pipe, which is what
  // bounds this kernel, once instead of twice. Copies of fewer records would be bound by their number (13 G a second).
  const bool bulk = levels <= kSplitBulkLevels;
  int tree = -1;                                 // whose splitters the tree holds
  SplitJob job = src.job(sh, b, tile);
  typename Src::Raw raw;
  src.load(sh, b, job, raw);
  for (;;) {
    if (tid < buckets) {
      s.count[tid] = 0;
      if (job.bucket != tree) {
        const int j = tid ? heap_rank(tid, levels) : 0;
        s.heap[tid] = tid && j < job.live ? Src::samples(sh, b, job.bucket)[j * kSplitOver] : ~0ull;           // ~0: above every key
      }
    }
    tree = job.bucket;
    uint64_t key[kSplitItems];
    src.keys(raw, key, b.status);
    __syncthreads();
    uint32_t at[kSplitItems];
#pragma unroll
    for (int t = 0; t < kSplitItems; ++t) at[t] = 1;
    for (int l = 0; l < levels; ++l)
#pragma unroll
      for (int t = 0; t < kSplitItems; ++t) at[t] = 2 * at[t] + (key[t] >= s.heap[at[t]] ? 1 : 0);
#pragma unroll
    for (int t = 0; t < kSplitItems; ++t) at[t] -= buckets;
    // Where entries come in key order the lanes fall into one bucket, and one of them counts for all.
    if (job.valid == kSplitTile && __all_sync(0xffffffffu, at[0] == __shfl_sync(0xffffffffu, at[0], 0))) {
#pragma unroll
      for (int t = 0; t < kSplitItems; ++t) {
        const uint32_t d = at[t];
        uint32_t rank = 0;
        if (__all_sync(0xffffffffu, d == __shfl_sync(0xffffffffu, d, 0))) {
          if (lane == 0) rank = atomicAdd(&s.count[d], 32u);
          rank = __shfl_sync(0xffffffffu, rank, 0) + lane;
        } else {
          rank = atomicAdd(&s.count[d], 1u);
        }
        at[t] = (d << 16) | rank;
      }
    } else {
#pragma unroll
      for (int t = 0; t < kSplitItems; ++t)
        if (t * kSplitThreads + tid < job.valid) at[t] = (at[t] << 16) | atomicAdd(&s.count[at[t]], 1u);
    }
    uint64_t val[kSplitItems];
#pragma unroll
    for (int t = 0; t < kSplitItems; ++t) val[t] = t * kSplitThreads + tid < job.valid ? src.value(raw, job, t) : 0;
    __syncthreads();
    const uint32_t mine = tid < buckets ? s.count[tid] : 0;
    uint32_t base = 0;
    if (mine) base = atomicAdd(Src::cursor(sh, b, job.bucket, tid), mine);    // not needed before the records lie in order
    if (tid < 32) {                              // where the buckets start in the tile: one warp, a row of buckets a lane
      const int per = buckets >> 5;              // both splits have at least 32 buckets
      uint32_t sum = 0;
      for (int i = 0; i < per; ++i) sum += s.count[lane * per + i];
      uint32_t run = sum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, run, off);
        if (lane >= off) run += x;
      }
      run -= sum;
      for (int i = 0; i < per; ++i) {
        s.start[lane * per + i] = run;
        run += s.count[lane * per + i];
      }
    }
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");            // the last tile's records have left
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kSplitItems; ++t)
      if (t * kSplitThreads + tid < job.valid) {
        const uint32_t d = at[t] >> 16, p = s.start[d] + (at[t] & 0xffffu);
        s.rec[p] = SplitRecord{key[t], val[t]};
        if (!bulk) s.bucket[p] = (uint16_t)d;
      }
    const SplitJob now = job;
    ++tile;
    if (tile < end) {
      job = src.job(sh, b, tile);
      src.load(sh, b, job, raw);
    }
    const bool room = base + mine <= cap;
    if (!room) atomicOr(b.status + kStatusOverflow, 1);
    const int64_t to = now.region0 + (int64_t)tid * cap + base;  // where bucket `tid`'s run goes
    if (bulk) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
      if (mine && room) {
        const uint32_t from = (uint32_t)__cvta_generic_to_shared(&s.rec[s.start[tid]]);
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(out + to), "r"(from), "r"(mine * 16u) : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      }
    } else {
      if (tid < buckets) s.delta[tid] = room ? to - s.start[tid] : INT64_MIN;
      __syncthreads();
#pragma unroll
      for (int t = 0; t < kSplitItems; ++t) {    // consecutive threads write a bucket's run
        const int p = t * kSplitThreads + tid;
        if (p < now.valid) {
          const int64_t dst = s.delta[s.bucket[p]] + p;
          if (dst >= 0) out[dst] = s.rec[p];
        }
      }
    }
    if (tile >= end) break;
  }
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");              // before the shared memory goes
}

// ---------------------------------------------------------------------------------------------- fine buckets
struct __align__(16) SplitPiece {                // between two samples: cell = (key - lo) >> shift, times scale
  uint64_t lo;
  float scale;
  int shift;
};

struct SplitSorted {                             // where step 5 writes
  uint64_t *keys;                                // kSplitKeys: the sorted keys; the values go to `val` in every form
  void *val;
  int32_t *pos;                                  // kSplitCsr: the row level's positions; kSplitCoordinates: level 0's two
  int32_t *crd[COMET_MAX_ORDER];                 // kSplitCsr: [1]; kSplitCoordinates: every level
};
constexpr int kSplitKeys = 0, kSplitCsr = 1, kSplitCoordinates = 2;

struct SortShared {
  uint64_t key[kSplitCap];
  uint64_t val[kSplitCap];
  SplitPiece piece[32];
  uint64_t heap[32];
  __align__(16) uint32_t start[kSplitCells + 4];   // counts, then where the cells start
  uint32_t warp[32];
  uint32_t before;
  int32_t moved;
  uint16_t cell[kSplitCap];
};

// The body for a bucket of at most STEPS * kSplitThreads entries.
template <int ORDER, class V, int FORM, int STEPS>
__device__ __forceinline__ void sort_bucket(const KeyLayout &k, const SplitShape &sh, const SplitBuffers &b, const SplitSorted &out, uint32_t bucket,
                                            int c, int f, int m) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  SortShared &s = *reinterpret_cast<SortShared *>(s_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t *counts = b.cursor2 + ((size_t)c << sh.k2);
  const uint64_t *samples = b.samples2 + (((size_t)c << sh.k2) + f) * kSplitOver;
  SplitRecord r[STEPS];
  const SplitRecord *rec = b.rec2 + (size_t)bucket * kSplitCap;
#pragma unroll
  for (int t = 0; t < STEPS; ++t) {
    const int i = t * kSplitThreads + tid;
    if (i < m) {
      const ulonglong2 two = __ldcs(reinterpret_cast<const ulonglong2 *>(rec + i));
      r[t] = SplitRecord{two.x, two.y};
    }
  }
  // the first position: entries of the fine buckets in front (at most 255)
  uint32_t front = tid < f ? counts[tid] : 0;
  if (front > kSplitCap) front = kSplitCap;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) front += __shfl_down_sync(0xffffffffu, front, off);
  if (lane == 0) s.warp[warp] = front;
  if (tid < 32) {                                // the pieces between the bucket's samples
    const bool last_fine = f + 1 >= (int)(b.fine_base[c + 1] - b.fine_base[c]);
    const uint64_t lo = tid == 0 && f == 0 ? coarse_bound(sh, b, c) : samples[tid];
    const uint64_t hi = tid == 31 && last_fine ? coarse_bound(sh, b, c + 1) : samples[tid + 1];
    const uint64_t most = hi > lo ? hi - lo - 1 : 0;
    SplitPiece p;
    p.lo = lo;
    p.shift = most >> 31 ? 33 - __clzll((long long)most) : 0;           // at most 31 bits are left
    p.scale = (float)kPieceCells / ((float)(uint32_t)(most >> p.shift) + 1.0f);
    s.piece[tid] = p;
    s.heap[tid] = tid ? samples[heap_rank(tid, 5)] : 0;
  }
  *reinterpret_cast<uint4 *>(&s.start[4 * tid]) = make_uint4(0, 0, 0, 0);
  if (tid == 0) s.moved = 0;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < kSplitThreads / 32 ? s.warp[lane] : 0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) w += __shfl_down_sync(0xffffffffu, w, off);
    if (lane == 0) s.before = w + b.coarse_start[c];
  }
  uint32_t at[STEPS];
#pragma unroll
  for (int t = 0; t < STEPS; ++t) {
    const int i = t * kSplitThreads + tid;
    if (i < m) {
      const uint64_t key = r[t].key;
      uint32_t h = 1;
#pragma unroll
      for (int l = 0; l < 5; ++l) h = 2 * h + (key >= s.heap[h] ? 1 : 0);
      h -= 32;
      const SplitPiece p = s.piece[h];
      int cell = (int)((float)(uint32_t)((key - p.lo) >> p.shift) * p.scale);      // grows with the key
      cell = (int)h * kPieceCells + (cell < kPieceCells - 1 ? cell : kPieceCells - 1);
      at[t] = ((uint32_t)cell << 16) | atomicAdd(&s.start[cell], 1u);
    }
  }
  __syncthreads();
  {
    static_assert(kSplitCells == 4 * kSplitThreads, "four cells a thread");
    const uint4 n4 = *reinterpret_cast<const uint4 *>(&s.start[4 * tid]);
    uint4 at4;
    const uint32_t four = n4.x + n4.y + n4.z + n4.w;
    uint32_t run = four;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, run, off);
      if (lane >= off) run += x;
    }
    if (lane == 31) s.warp[warp] = run;
    __syncthreads();
    at4.x = run - four + __reduce_add_sync(0xffffffffu, lane < warp ? s.warp[lane] : 0);
    at4.y = at4.x + n4.x; at4.z = at4.y + n4.y; at4.w = at4.z + n4.z;
    *reinterpret_cast<uint4 *>(&s.start[4 * tid]) = at4;
    if (tid == 0) s.start[kSplitCells] = m;
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < STEPS; ++t) {
    const int i = t * kSplitThreads + tid;
    if (i < m) {
      const uint32_t cell = at[t] >> 16, p = s.start[cell] + (at[t] & 0xffffu);
      s.key[p] = r[t].key;
      s.val[p] = r[t].val;
      s.cell[p] = (uint16_t)cell;
    }
  }
  __syncthreads();
  const uint32_t before = s.before;
  int moved = 0;                                 // the places are all different exactly if their sum is that of 0 .. m - 1
#pragma unroll
  for (int t = 0; t < STEPS; ++t) {        // an entry's place: the smaller keys of its cell
    const int p = t * kSplitThreads + tid;
    if (p < m) {
      const uint64_t key = s.key[p];
      const uint32_t cell = s.cell[p];
      uint32_t q = s.start[cell];
      const uint32_t end = s.start[cell + 1];
      for (uint32_t j = q; j < end; ++j) q += s.key[j] < key ? 1 : 0;
      moved += (int)q - p;
      if (FORM == kSplitCsr) at[t] = (q << 16), r[t].key = key;
      if (sizeof(V) == 8) __stcs(static_cast<unsigned long long *>(out.val) + before + q, (unsigned long long)s.val[p]);
      else __stcs(static_cast<uint32_t *>(out.val) + before + q, (uint32_t)s.val[p]);
      if (FORM == kSplitKeys) out.keys[before + q] = key;
      if (FORM == kSplitCoordinates) {
#pragma unroll
        for (int l = 0; l < ORDER; ++l) __stcs(out.crd[l] + before + q, (int32_t)((key >> k.shift[l]) & ((1ull << k.bits[l]) - 1)));
      }
      if (FORM == kSplitCsr) __stcs(out.crd[1] + before + q, (int32_t)(key & ((1ull << k.bits[1]) - 1)));
    }
  }
  moved = __reduce_add_sync(0xffffffffu, moved);
  if (lane == 0 && moved) atomicAdd(&s.moved, moved);
  __syncthreads();
  const bool equal = s.moved != 0;                                        // equal keys took one place, another one is free
  if (tid == 0 && equal) atomicOr(b.status + kStatusDuplicate, 1);
  if (FORM != kSplitCsr || equal) return;
  uint32_t *rows = reinterpret_cast<uint32_t *>(s.val);                   // the rows in order, over the values
#pragma unroll
  for (int t = 0; t < STEPS; ++t)
    if (t * kSplitThreads + tid < m) rows[at[t] >> 16] = (uint32_t)(r[t].key >> k.shift[0]);
  __syncthreads();
#pragma unroll
  for (int t = 0; t < STEPS; ++t) {
    const int p = t * kSplitThreads + tid;
    if (p < m && p > 0) {
      const uint32_t row = rows[p], prev = rows[p - 1];
      for (uint32_t x = prev + 1; x <= row; ++x) out.pos[x] = (int32_t)(before + p);
    }
  }
  if (tid == 0) b.edges[bucket] = make_uint4(rows[0], rows[m - 1], before, m);
}

template <int ORDER, class V, int FORM>
__global__ void __launch_bounds__(kSplitThreads, 3) split_sort_kernel(KeyLayout k, SplitShape sh, SplitBuffers b, SplitSorted out) {
  const uint32_t bucket = blockIdx.x;
  if (FORM == kSplitCoordinates && bucket == 0 && threadIdx.x == 0) { out.pos[0] = 0; out.pos[1] = (int32_t)sh.n; }
  if (bucket >= b.totals[1]) return;
  if (b.status[kStatusOverflow] | b.status[kStatusRange]) return;      // records may be missing, or their rows beyond the matrix
  const int c = b.fine_map[bucket];
  const int f = bucket - b.fine_base[c];
  const uint32_t got = b.cursor2[((size_t)c << sh.k2) + f];
  const int m = got < kSplitCap ? (int)got : kSplitCap;
  if (m == 0) {
    if (FORM == kSplitCsr && threadIdx.x == 0) b.edges[bucket] = make_uint4(0, 0, 0, 0);
    return;
  }
  // most buckets have at most four entries a thread: their loops are half as long
  if (m <= 4 * kSplitThreads) sort_bucket<ORDER, V, FORM, 4>(k, sh, b, out, bucket, c, f, m);
  else sort_bucket<ORDER, V, FORM, (kSplitCap + kSplitThreads - 1) / kSplitThreads>(k, sh, b, out, bucket, c, f, m);
}

// CSR: the rows that start between two fine buckets, and those behind the last entry.
__global__ void split_csr_edges_kernel(SplitBuffers b, int64_t n, int64_t rows, int32_t *__restrict__ pos0, int32_t *__restrict__ pos) {
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, threads = (int64_t)gridDim.x * blockDim.x;
  const int64_t fines = b.totals[1];
  if (b.status[kStatusOverflow] | b.status[kStatusRange] | b.status[kStatusDuplicate]) return;    // not every bucket has edges
  if (tid == 0) pos0[0] = (int32_t)rows;
  for (int64_t i = tid; i < fines; i += threads) {
    const uint4 e = b.edges[i];
    if (!e.w) continue;
    int64_t prev = i - 1;
    while (prev >= 0 && !b.edges[prev].w) --prev;
    const int64_t from = prev >= 0 ? (int64_t)b.edges[prev].y : -1;
    for (int64_t x = from + 1; x <= (int64_t)e.x; ++x) pos[x] = (int32_t)e.z;
  }
  int64_t last = fines - 1;
  while (last >= 0 && !b.edges[last].w) --last;
  const int64_t from = last >= 0 ? (int64_t)b.edges[last].y : -1;
  for (int64_t x = from + 1 + tid; x <= rows; x += threads) pos[x] = (int32_t)n;
}

// ---------------------------------------------------------------------------------------------- host
static size_t split_layout(const SplitShape &sh, char *block, SplitBuffers *b) {
  size_t used = 0;
  auto take = [&](size_t bytes) { char *p = block + used; used += align_up(bytes, 256); return p; };
  const size_t f1 = (size_t)1 << sh.k1, all = f1 << sh.k2;
  b->cursor1 = (uint32_t *)take(f1 * kSplitCursorStride * 4);
  b->cursor2 = (uint32_t *)take(all * 4);
  b->drawn = (uint64_t *)take(f1 * kSplitOver * 8);
  b->samples1 = (uint64_t *)take(f1 * kSplitOver * 8);
  b->samples2 = (uint64_t *)take(all * kSplitOver * 8);
  b->coarse_start = (uint32_t *)take((f1 + 1) * 4);
  b->fine_base = (uint32_t *)take((f1 + 1) * 4);
  b->tile_map = (uint4 *)take((size_t)sh.tile_max * 16);
  b->fine_map = (uint32_t *)take((size_t)sh.fine_max * 4);
  b->totals = (uint32_t *)take(8);
  b->edges = (uint4 *)take((size_t)sh.fine_max * 16);
  b->rec1 = (SplitRecord *)take(f1 * sh.cap1 * 16);
  b->rec2 = (SplitRecord *)take((size_t)sh.fine_max * kSplitCap * 16);
  return used;
}

// Small inputs have a launch of their own (pack_small.cu), which is as fast at 400,000 to 600,000 entries (97 against 97 us for
// a matrix, 121 against 130 for a CSF tensor) and slower from there on (620,000 entries 142 against 106; 700,000 to CSF 165
// against 145). At most 512 coarse buckets of 160 fine ones fit.
bool pack_split_applies(int order, int total_bits, int64_t n) {
  int64_t least = 600000;
  if (const char *e = getenv("COMET_PACK_SPLIT")) least = e[0] == '0' ? INT64_MAX : 1;      // tests: "1" takes this path on any size, "0" never
  return order >= 2 && total_bits >= 1 && n >= least && n <= 512ll * 160 * kSplitMean;
}

size_t pack_split_bytes(int64_t n) {
  SplitBuffers b;
  return split_layout(split_shape(n, 0), nullptr, &b);
}

static size_t split_shared(int levels) { return levels <= kSplitBulkLevels ? offsetof(SplitShared, delta) : sizeof(SplitShared); }

template <class K>
static comet_status_t big_shared(Context *ctx, K kernel, size_t bytes) {
  COMET_CUDA_TRY(ctx, cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  return COMET_OK;
}

template <int ORDER, class V, int FORM>
static comet_status_t launch_sort(Context *ctx, const KeyLayout &k, const SplitShape &sh, const SplitBuffers &b, const SplitSorted &out,
                                  cudaStream_t s) {
  const comet_status_t st = big_shared(ctx, split_sort_kernel<ORDER, V, FORM>, sizeof(SortShared));
  if (st != COMET_OK) return st;
  split_sort_kernel<ORDER, V, FORM><<<(unsigned)sh.fine_max, kSplitThreads, sizeof(SortShared), s>>>(k, sh, b, out);
  COMET_LAUNCH_CHECK(ctx);
  return COMET_OK;
}

template <int ORDER>
static comet_status_t run_split(Context *ctx, const CoordPtrs &c, const KeyLayout &k, const void *val, bool f32, int64_t n, char *tmp,
                                const LevelOut *direct, int form, PackSplitSorted *sorted, cudaStream_t s) {
  const SplitShape sh = split_shape(n, k.total_bits);
  SplitBuffers b;
  split_layout(sh, tmp, &b);
  b.status = ctx->d_status;
  const unsigned f1 = 1u << sh.k1;
  uintptr_t low = reinterpret_cast<uintptr_t>(val);
  for (int l = 0; l < ORDER; ++l) low |= reinterpret_cast<uintptr_t>(c.p[l]);
  const bool wide = (low & 15) == 0;
  const size_t coarse_bytes = (size_t)f1 * kSplitOver * 8, fine_bytes = kMostSamples * 8;
  comet_status_t st = big_shared(ctx, split_rank_samples_kernel, coarse_bytes);
  if (st == COMET_OK) st = big_shared(ctx, split_sample_fine_kernel, fine_bytes);
  if (st == COMET_OK) st = big_shared(ctx, split_kernel<SplitCoo<ORDER>>, sizeof(SplitShared));
  if (st == COMET_OK) st = big_shared(ctx, split_kernel<SplitRec>, sizeof(SplitShared));
  if (st != COMET_OK) return st;
  split_sample_coarse_kernel<ORDER><<<(unsigned)ceil_div((int64_t)f1 * kSplitOver, kSplitThreads), kSplitThreads, 0, s>>>(c, k, sh, b);
  split_rank_samples_kernel<<<kSmCount, kSampleThreads, coarse_bytes, s>>>(sh, b);
  const unsigned ctas = 2 * kSmCount;
  split_kernel<SplitCoo<ORDER>><<<ctas, kSplitThreads, split_shared(sh.k1), s>>>(SplitCoo<ORDER>{c, k, val, f32, wide}, sh, b, sh.k1, (uint32_t)sh.cap1, b.rec1);
  split_sample_fine_kernel<<<f1 + 1, kSampleThreads, fine_bytes, s>>>(sh, b);
  split_kernel<SplitRec><<<ctas, kSplitThreads, split_shared(sh.k2), s>>>(SplitRec{}, sh, b, sh.k2, kSplitCap, b.rec2);
  COMET_LAUNCHED(ctx, 5);
  SplitSorted out{};
  if (form == kSplitKeys) {                      // over the first split's records, which nothing reads any more
    sorted->keys = out.keys = reinterpret_cast<uint64_t *>(b.rec1);
    sorted->val = out.val = out.keys + align_up((size_t)n + 1, 32);
  } else {
    out.val = direct->val;
    out.pos = form == kSplitCsr ? direct->pos[1] : direct->pos[0];
    for (int l = 0; l < ORDER; ++l) out.crd[l] = direct->crd[l];
  }
  if (form == kSplitCsr) {
    if constexpr (ORDER == 2) {
      st = f32 ? launch_sort<2, float, kSplitCsr>(ctx, k, sh, b, out, s) : launch_sort<2, double, kSplitCsr>(ctx, k, sh, b, out, s);
      if (st != COMET_OK) return st;
      split_csr_edges_kernel<<<kSmCount, 256, 0, s>>>(b, n, direct->dim0, direct->pos[0], direct->pos[1]);
      COMET_LAUNCH_CHECK(ctx);
    }
    return COMET_OK;
  }
  if (form == kSplitCoordinates)
    return f32 ? launch_sort<ORDER, float, kSplitCoordinates>(ctx, k, sh, b, out, s)
               : launch_sort<ORDER, double, kSplitCoordinates>(ctx, k, sh, b, out, s);
  return f32 ? launch_sort<ORDER, float, kSplitKeys>(ctx, k, sh, b, out, s) : launch_sort<ORDER, double, kSplitKeys>(ctx, k, sh, b, out, s);
}

comet_status_t pack_split_sort(Context *ctx, int order, const CoordPtrs &c, const KeyLayout &k, const LevelPlan &plan, const void *val,
                               int dtype, int64_t n, char *tmp, const LevelOut *direct, PackSplitSorted *sorted, cudaStream_t s) {
  const bool f32 = dtype == COMET_F32;
  const int form = !direct ? kSplitKeys : plan.attr[0] == COMET_D ? kSplitCsr : kSplitCoordinates;
  if (order == 2) return run_split<2>(ctx, c, k, val, f32, n, tmp, direct, form, sorted, s);
  if (order == 3) return run_split<3>(ctx, c, k, val, f32, n, tmp, direct, form, sorted, s);
  return run_split<4>(ctx, c, k, val, f32, n, tmp, direct, form, sorted, s);
}

}  // namespace comet

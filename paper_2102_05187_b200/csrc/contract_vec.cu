// Segment-gather contractions with a dense matrix operand: SpMM, TTM (the SpMM/SpTTM definitions of
// the paper's Sparse Tensor Operations subsection). Both are "for every leaf entry p of segment s:
// out[s, :] += val[p] * B[crd[p], :]" where a segment is a CSR row (SpMM) or a CSF fiber (TTM).
//
// Work split (B200): the merge list of segment-end markers and leaf positions is cut into tiles of a
// fixed number of items, one tile per WORKER (a group of LPN lanes of a warp, see walk.cuh). A worker
// walks its tile sequentially with a rolling window of row gathers in flight, stores every segment
// that ENDS inside its tile with plain vector stores (so every output row is written exactly once,
// without a memset), and hands the partial sum of the segment it stops in to a carry slot. A second
// small kernel adds the carries of earlier tiles onto the stored rows in tile order, which makes the
// result deterministic (no atomics anywhere).
#include "common.cuh"
#include "kernels.cuh"
#include "walk.cuh"
#include "spmm_heavy.cuh"

#ifndef COMET_PF_GATHER
#define COMET_PF_GATHER 4      // row gathers in flight per worker (SpMM, TTM); measured best with 4 CTAs/SM
#endif
#ifndef COMET_MINB_GATHER
#define COMET_MINB_GATHER 4    // CTAs per SM the register budget is held to (64 registers)
#endif

namespace comet {

struct SegGatherArgs {
  const int32_t *seg_end;   // M entries: leaf position where segment s ends (= pos + 1)
  const int32_t *crd;       // N leaf coordinates (row index into B)
  const void *val;          // N values (T)
  int64_t M, N;
  const void *B;            // dense operand (T), already offset to this launch's first column
  int64_t ldb;
  void *C;                  // output rows (T), already offset to this launch's first column
  int64_t ldc;
  const int32_t *out_row;   // NULL: segment s -> row s. Else segment s -> row out_row[s] (ascending); the rows in between
  int64_t out_rows;         //   (and up to out_rows) hold zeros already or are cleared by the CTAs from gap_from on
  int64_t gap_from;
  int32_t R;                // columns handled by this launch
  bool wide_store;          // ragged shapes: rows of C take 16-byte stores
  int32_t tile_items;
  int64_t num_tiles;
  double *carry_val;        // num_tiles x carry_ld
  int32_t *carry_seg;       // num_tiles: segment the carry belongs to, -1 if none
  int32_t carry_ld;
  const int32_t *part;      // num_tiles + 1 merge-path splits (segments in front of each tile boundary), or NULL
  int32_t own_len;          // segments of at most this many entries are processed whole by the tile of their end marker
  int32_t skip_len;         // > 0: segments of at least this many entries are somebody else's (the long-row
                            //      path of SpMM): neither walked nor stored here. Never below tile_items.
};

// Where the rows of C go: segment s to row s, or through out_row. Two kernels, not a test, as the closing of a segment sits in
// the body that is unrolled for every entry of a chunk.
constexpr int kRowsAll = 0, kRowsMapped = 1;

// What the walker does with one leaf entry: close the segments that end in front of it, accumulate.
template <class T, int LPN, int CPL, int VEC, bool RAGGED, int ROWS, bool PASS_THROUGH = false>
struct SegGatherPolicy {
  using L = Lanes<T, LPN, CPL, VEC, RAGGED>;
  // PASS_THROUGH: the general rows beside the long ones, which come from DRAM: eight rows in flight (walk_tile_async)
  static constexpr int kPF = PASS_THROUGH && CPL == 1 ? 2 * COMET_PF_GATHER : COMET_PF_GATHER;
  static constexpr bool kAux = false;
  // Ragged fp32 rows end in up to four scalar stores per lane, too much code for one copy per entry of the chunk: with the
  // chunk unrolled the kernel waits for instructions (30 M entries, R = 50: 519 us unrolled, 475 rolled).
  static constexpr bool kFullUnroll = !(RAGGED && sizeof(T) == 4);
  // one copy of the unrolled body where the chunk is long (instruction cache; measured: SpMM config 2 -4 %); the
  // narrow shapes have short tiles of short chunks, where the slower rolled tail costs more than it saves (TTM +5 %)
  static constexpr bool kRolledTail = LPN >= 16;
  struct Slot { T r[CPL][VEC]; };

  const SegGatherArgs &a;
  const L &ln;
  const char *bcol;         // this lane's piece 0 of row 0 of B
  double acc[CPL][VEC];
  // The segment state is three words (the rest is recomputed where a segment closes): registers are what the
  // window of gathers in flight is made of.
  int32_t seg;              // the open segment
  int32_t base, rel_end;    // chunk base; where the open segment ends, relative to it (negative: no segment left)
  uint64_t pass;            // PASS_THROUGH: L2 evict-first policy of the gathers (the other role's block of B stays)

  __device__ __forceinline__ SegGatherPolicy(const SegGatherArgs &args, const L &lanes, int64_t i0, int32_t j0)
      : a(args), ln(lanes), seg((int32_t)i0), base(j0) {
    ln.zero(acc);
    if (PASS_THROUGH) pass = l2_policy_evict_first();
    bcol = reinterpret_cast<const char *>(static_cast<const T *>(a.B) + ln.load_col());
    rel_end = end_of_open();
  }
  __device__ __forceinline__ int32_t end_of_open() const {
    return seg < a.M ? __ldg(a.seg_end + seg) - base : (int32_t)0x80000000 / 2;
  }
  __device__ __forceinline__ int64_t segment() const { return seg; }
  __device__ __forceinline__ void fetch(int32_t j, Entry16 &e, int32_t &) const {
    e.v = (double)ld_stream(static_cast<const T *>(a.val) + j);
    e.a = ld_stream(a.crd + j);
  }
  __device__ __forceinline__ void fetch_async(int32_t j, uint32_t entry, bool there) const {
    if (sizeof(T) == 8) copy_async8(entry, static_cast<const T *>(a.val) + j, there);
    else copy_async4(entry, static_cast<const T *>(a.val) + j, there);
    copy_async4(entry + 8, a.crd + j, there);
  }
  __device__ __forceinline__ void settle(uint32_t entry) const {       // values are read as doubles
    if (sizeof(T) == 4) sts_f64(entry, (double)__int_as_float(lds_s32(entry)));
  }
  __device__ __forceinline__ void prefetch(int32_t c, int32_t, Slot &s) const {
    const T *row = reinterpret_cast<const T *>(bcol + (int64_t)c * (int32_t)(a.ldb * sizeof(T)));
    if (PASS_THROUGH) ln.gather_hint(row, s.r, pass);
    else ln.gather(row, s.r);
  }
  __device__ __forceinline__ void begin_chunk(int32_t b) { rel_end -= b - base; base = b; }

  __device__ __forceinline__ void flush() {      // stores the open segment
    T *cmat = static_cast<T *>(a.C) + ln.col0;
    // (asking for the row, or the next end, when the segment opens takes the registers that the window needs: this kernel
    // alone 65 -> 76 us on 2 M entries, R = 16; TTM of 30 M 345 -> 399)
    const int64_t row = ROWS == kRowsMapped ? (int64_t)__ldg(a.out_row + seg) : (int64_t)seg;
    ln.store_row(cmat + row * a.ldc, acc);
    ln.zero(acc);
    ++seg;
    rel_end = end_of_open();
  }
  __device__ __forceinline__ void consume(int q, double v, int32_t, Slot &s) {
    while (rel_end == q) flush();              // segments (possibly empty ones) that end in front of this leaf
    ln.fma_rows(v, s.r, acc);
  }
};

// Clears those of kGapRows rows of C that no segment owns (block b: rows b * kGapRows and on). The stored rows of the block are
// marked in shared memory, then consecutive threads clear consecutive pieces of the others: about the same work for
// every block wherever the empty rows lie. As CTAs of the gather kernel, whose rows are other ones, this costs no launch.
// When the workers filled the rows in front of each segment that they closed, the code for that sat in every entry of the
// unrolled chunk, and a tile with a long gap held its workers up: DCSR, power-law rows, all of them stored, fp64, 5.6 M entries,
// R = 32 435 us, as here 130; fp32, 4.5 M, R = 31 196 and 135; 2 M entries in 491,000 of 500,000 rows, R = 16 98 and 59.
constexpr int kGapRows = 1024;         // 256 / 512 / 1,024 / 2,048 rows: 6.6 M entries in 2.1 M of 2.2 M rows, fp32, R = 31 393 / 375 / 355 / 434 us
template <class T>
__device__ __forceinline__ void gap_role(const SegGatherArgs &a, int64_t block, unsigned char *smem) {
  static_assert(kGapRows % kBlockThreads == 0 && kGapRows / 32 < kBlockThreads, "");
  uint32_t *const bits = reinterpret_cast<uint32_t *>(smem), *const empties = bits + kGapRows / 32;
  uint16_t *const empty = reinterpret_cast<uint16_t *>(empties + 1);        // the empty rows, in any order
  const int64_t r0 = block * kGapRows;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x <= kGapRows / 32) bits[threadIdx.x] = 0;                  // and their number
  int64_t lo = 0, hi = a.M;                                // the first segment whose row is r0 or behind it
  while (lo < hi) {
    const int64_t stride = (hi - lo + 31) / 32;
    const int64_t q = lo + (int64_t)lane * stride + stride - 1;
    const int full = __popc(__ballot_sync(0xffffffffu, q < hi && __ldg(a.out_row + q) < r0));
    lo += (int64_t)full * stride;
    const int64_t cap = lo + stride - 1;
    if (cap < hi) hi = cap;
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < kGapRows / kBlockThreads; ++t) {     // rows are distinct: at most kGapRows of them lie in the block
    const int64_t mine = lo + t * kBlockThreads + threadIdx.x;
    const int64_t at = mine < a.M ? (int64_t)__ldg(a.out_row + mine) - r0 : kGapRows;
    if (at < kGapRows) atomicOr(&bits[at >> 5], 1u << (at & 31));
  }
  __syncthreads();
  const int rows = (int)(a.out_rows - r0 < kGapRows ? a.out_rows - r0 : kGapRows);
  constexpr int PER = 16 / sizeof(T);
  const bool wide = a.wide_store && a.R % PER == 0;
  const int width = wide ? a.R / PER : a.R;
  T *const C = static_cast<T *>(a.C) + r0 * a.ldc;
  for (int r = threadIdx.x; r < rows; r += kBlockThreads)
    if (!((bits[r >> 5] >> (r & 31)) & 1u)) empty[atomicAdd(empties, 1u)] = (uint16_t)r;
  __syncthreads();
  const int work = (int)*empties * width;
  for (int i = threadIdx.x; i < work; i += kBlockThreads) {
    const int e = i / width, c = i - e * width, r = empty[e];
    if (wide) __stcs(reinterpret_cast<int4 *>(C + (int64_t)r * a.ldc) + c, make_int4(0, 0, 0, 0));
    else __stcs(C + (int64_t)r * a.ldc + c, (T)0);
  }
}

// HEAVY: the first h.heavy_ctas CTAs of the grid work on the long rows of an SpMM (spmm_heavy.cuh) while the
// others walk the general tiles and skip those rows. The two roles are bound by different things (the long rows
// by the L2 -> L1 fill rate, the rest by DRAM latency), so sharing the SMs between them is faster than running
// one after the other.
template <class T, int LPN, int CPL, int VEC, bool RAGGED, int ROWS, bool HEAVY>
__global__ void __launch_bounds__(kBlockThreads, (CPL * VEC * sizeof(T) <= 16 ? COMET_MINB_GATHER : 2))
seg_gather_kernel(const SegGatherArgs a, const HeavyArgs h) {
  using L = Lanes<T, LPN, CPL, VEC, RAGGED>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (HEAVY && (int)blockIdx.x < h.heavy_ctas) {
    heavy_role<T, LPN, CPL, VEC>(h, smem_raw);
    return;
  }
  if (ROWS == kRowsMapped && (int64_t)blockIdx.x >= a.gap_from) {
    gap_role<T>(a, (int64_t)blockIdx.x - a.gap_from, smem_raw);
    return;
  }
  const int worker = threadIdx.x / LPN;
  const int64_t tile = (int64_t)(blockIdx.x - (HEAVY ? h.heavy_ctas : 0)) * L::kWorkers + worker;
  if (tile >= a.num_tiles) return;                       // whole groups leave together
  const uint32_t smem = smem_u32(smem_raw) + worker * (HEAVY ? AsyncRing<L>::kWorkerBytes : RingLayout<L, false>::kWorkerBytes);
  const L ln(a.R, a.wide_store);
  if (tile == 0) clear_piece_counts(a.carry_seg, a.num_tiles, ln.g, LPN);

  const int64_t total = a.M + a.N;
  const int64_t d0 = tile * a.tile_items;
  const int64_t d1 = (d0 + a.tile_items < total) ? d0 + a.tile_items : total;
  // the splits come from the partition kernel when there is one: a worker is sequential, and two dependent
  // searches at the head of every tile are a sizeable part of a short tile
  int64_t i0 = a.part ? (int64_t)__ldg(a.part + tile) : merge_path_segments_coop<LPN>(a.seg_end, a.M, a.N, d0, ln.g, ln.mask);
  const int64_t i1 = a.part ? (int64_t)__ldg(a.part + tile + 1) : merge_path_segments_coop<LPN>(a.seg_end, a.M, a.N, d1, ln.g, ln.mask);
  int32_t j0 = (int32_t)(d0 - i0), j1 = (int32_t)(d1 - i1);
  if (a.skip_len > 0) {
    // A long segment holds more entries than a tile, so it can only be the one open at the tile's start or the
    // one open at its end. Its entries are left out; its end marker (if it is in this tile) stores nothing.
    if (i0 < a.M) {
      const int32_t end0 = __ldg(a.seg_end + i0);
      const int32_t start0 = i0 > 0 ? __ldg(a.seg_end + i0 - 1) : 0;
      if (end0 - start0 >= a.skip_len) {
        if (i0 >= i1) {                                      // the whole tile lies inside the long segment
          if (ln.g == 0) a.carry_seg[tile] = -1;
          return;
        }
        i0 += 1;
        j0 = end0;
      }
    }
    if (i1 < a.M) {
      const int32_t start1 = i1 > 0 ? __ldg(a.seg_end + i1 - 1) : 0;
      if (__ldg(a.seg_end + i1) - start1 >= a.skip_len && start1 < j1) j1 = start1 > j0 ? start1 : j0;
    }
  }

  // A segment of at most `own_len` entries belongs wholly to the tile that holds its end marker: the tile
  // in front leaves the segment's first entries out and this one takes them, so such a segment needs no carry
  // (and no fix-up work). Both tiles look at the same segment and decide alike; longer segments are split as
  // before. The limit is a quarter of a tile, so that tiles stay within 25 % of their nominal size.
  // Measured: config 4 TTM 416 -> 399 us with any limit from an eighth of a tile to a whole one. Not done beside
  // the long-row role (SpMM config 2: 1017 us without, 1020 / 1026 / 1041 / 1079 us with an eighth / a quarter / half
  // a tile / a whole tile: its rows of a few hundred entries make the tiles uneven, which costs more than their
  // carries did).
  if (!HEAVY) {
    if (i0 < a.M) {
      const int32_t start0 = i0 > 0 ? __ldg(a.seg_end + i0 - 1) : 0;
      if (__ldg(a.seg_end + i0) - start0 <= a.own_len && start0 < j0) j0 = start0;
    }
    if (i1 < a.M) {
      const int32_t start1 = i1 > 0 ? __ldg(a.seg_end + i1 - 1) : 0;
      if (__ldg(a.seg_end + i1) - start1 <= a.own_len && start1 < j1) j1 = start1 > j0 ? start1 : j0;
    }
  }

  SegGatherPolicy<T, LPN, CPL, VEC, RAGGED, ROWS, HEAVY> p(a, ln, i0, j0);
  if constexpr (HEAVY) walk_tile_async(ln, p, j0, j1, smem);
  else walk_tile(ln, p, j0, j1, smem);
  while (p.segment() < i1) p.flush();                    // end markers that close the tile

  // leaf entries of a segment that ends in a later tile: the open segment starts in front of the tile's end
  const int64_t seg = p.segment();
  const int32_t open_from = seg > 0 ? __ldg(a.seg_end + seg - 1) : 0;
  const bool carry = seg < a.M && (open_from > j0 ? open_from : j0) < j1;
  if (ln.g == 0) a.carry_seg[tile] = carry ? (int32_t)seg : -1;
  if (carry) ln.store_carry(a.carry_val + tile * a.carry_ld + ln.col0, p.acc);
}

// Adds the carries onto the stored rows. The tiles that stopped inside one segment are consecutive (a run); the sum of
// a run is added to the segment's row, which has no other writer by now. One thread per tile and pair of columns: the
// threads at the head of a run add it up, several tiles in flight. What bounds this is latency, and a run of thousands of
// tiles (a slice that holds most of a tensor) would be a serial chain: a run of more than run_short() tiles is therefore
// added by the whole CTA of its head, and (cut) runs are cut at the multiples of kRunPiece tiles behind which they go on for
// kRunSpare tiles and more: a piece's sum stays in the slot of its first tile, and the CTA that finishes the last piece of a
// run adds the pieces (each counts itself done; none waits). Every order is fixed. Finishing a piece costs about 4 us, and
// some run crosses a multiple almost always: with short runs cut too, MTTKRP of 90,000 entries (CSF, R = 6) took 31.3 us
// instead of 26.7, of 78,000 (COO, R = 5) 20.7 instead of 15.8. Measured, runs followed by one thread -> as here: 0.85 M
// entries, R = 4, 60 % of them in one slice 918 -> 84 us (whole CSF MTTKRP); 14.9 M entries, R = 32 3.05 -> 0.39 ms (COO);
// 100 M entries, heaviest slice 0.5 % 2.90 -> 2.84 ms.
// Tiles up to which a thread follows a run. Beyond, the run takes its CTA about 3 us, and a CTA takes the runs of its tiles one
// after the other, while the threads follow theirs side by side, 0.7 us per eight tiles: the narrower the rows, the more
// tiles (and runs) a CTA has. A power-law matrix of 19.5 M entries times a vector: 135 us with 12 for every width, 106 us
// when the limit grows with the tiles per CTA.
__device__ __forceinline__ int32_t run_first(int32_t R) { return R == 1 ? 8 : 4; }     // tiles read at once to begin with
__device__ __forceinline__ int32_t run_short(int32_t R, int32_t tiles) {
  return run_first(R) + (tiles >= 128 ? 96 : tiles >= 32 ? 32 : tiles >= 16 ? 24 : 8);
}

struct FixupArgs {
  double *carry_val;
  const int32_t *carry_seg;
  int32_t num_tiles;
  int32_t R, carry_ld;
  void *C;
  int64_t ldc;
  const int32_t *out_row;
  int32_t *done;                                 // per multiple of kRunPiece: pieces of the run first cut there that are summed
                                                 // (zero at the start; NULL: runs are not cut)
};

constexpr int32_t kRunSpare = 128;
// Whether a run of segment `seg` that crosses tile t, a multiple of kRunPiece, is cut there. (The tiles in between are the
// run's too.)
__device__ __forceinline__ bool run_cut_at(const FixupArgs &f, int64_t t, int32_t seg) {
  return t + kRunSpare < f.num_tiles && __ldg(f.carry_seg + t + kRunSpare) == seg;
}

template <class T>
__device__ __forceinline__ void add_to_row(const FixupArgs &f, int32_t seg, int32_t c, double sum) {
  const int64_t row = f.out_row ? (int64_t)__ldg(f.out_row + seg) : (int64_t)seg;
  T *const dst = static_cast<T *>(f.C) + row * f.ldc + c;
  *dst = (T)((double)*dst + sum);
}

// The sum of the slots first, first + step, ... (count of them), over all threads of the CTA: group g of the 256 / R
// groups of R threads takes slots g, g + G, ..., the groups' sums are added in group order. Valid for threads below R.
__device__ __forceinline__ double cta_slot_sum(const FixupArgs &f, int64_t first, int64_t step, int32_t count, double *s_part) {
  const int32_t G = kBlockThreads / f.R;
  const int32_t g = threadIdx.x / f.R, c = threadIdx.x - g * f.R;
  double sum = 0.0;
  if (g < G) {
    const double *src = f.carry_val + first * f.carry_ld + c;
    const int64_t stride = step * f.carry_ld;
    for (int32_t q = g; q < count; q += 8 * G) {           // eight slots in flight, the last ones guarded
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = q + u * G < count ? __ldcg(src + (int64_t)(q + u * G) * stride) : 0.0;
#pragma unroll
      for (int u = 0; u < 8; ++u) sum += v[u];
    }
  }
  __syncthreads();
  s_part[threadIdx.x] = sum;
  __syncthreads();
  sum = 0.0;
  if (threadIdx.x < f.R)
    for (int32_t x = 0; x < G; ++x) sum += s_part[x * f.R + threadIdx.x];
  return sum;
}

// A part of a cut run is in its slot (tile `first`, written by threads of this CTA): counts it, and if it was the last part
// of the run adds them all up. A run of `pieces` cuts has pieces + 1 parts: its head's and one from every cut on.
template <class T>
__device__ __forceinline__ void finish_piece(const FixupArgs &f, int32_t first, int32_t seg, double *s_part, int32_t *s_old) {
  auto cut_at = [&](int64_t m) {                 // the run is cut at multiple m
    const int64_t t = m * kRunPiece;
    return m > 0 && run_cut_at(f, t, seg) && __ldg(f.carry_seg + t - 1) == seg;
  };
  __threadfence();
  __syncthreads();
  const int32_t here = first / kRunPiece;
  int32_t back = 0, ahead = 0, more;
  do {                                           // cuts at `here` and below, and above
    more = __syncthreads_count(cut_at((int64_t)here - back - (int32_t)threadIdx.x));
    back += more;
  } while (more == kBlockThreads);
  do {
    more = __syncthreads_count(cut_at((int64_t)here + 1 + ahead + threadIdx.x));
    ahead += more;
  } while (more == kBlockThreads);
  // a head that sits on a multiple is no cut itself; a head inside a piece sees the cuts above it only
  const int32_t m1 = here + 1 - back, pieces = back + ahead;
  if (threadIdx.x == 0) *s_old = atomicAdd(f.done + m1, 1);
  __syncthreads();
  const bool last = *s_old == pieces;
  __syncthreads();
  if (!last) return;
  __threadfence();
  const int32_t second = m1 * kRunPiece;
  int32_t lead = 0;                              // tiles of the head's part
  do {
    const int32_t t = second - 1 - lead - (int32_t)threadIdx.x;
    more = __syncthreads_count(t >= 0 && __ldg(f.carry_seg + t) == seg);
    lead += more;
  } while (more == kBlockThreads);
  const double sum = cta_slot_sum(f, second, kRunPiece, pieces, s_part);
  if (threadIdx.x < f.R)
    add_to_row<T>(f, seg, threadIdx.x, __ldcg(f.carry_val + (int64_t)(second - lead) * f.carry_ld + threadIdx.x) + sum);
  __syncthreads();
}

// `block` of fixup_blocks() CTAs: a thread per tile and pair of columns (half as many CTAs as with a column each: 27 ->
// 24 us for 37,000 tiles of 64 columns). LONG: long runs are possible.
__host__ __device__ __forceinline__ int32_t fixup_tiles(int32_t R) { return kBlockThreads / ((R + 1) / 2); }   // per CTA

template <class T, bool LONG>
__device__ __forceinline__ void carry_fixup_role(const FixupArgs &f, int64_t block) {
  const int32_t per = (f.R + 1) / 2, G = fixup_tiles(f.R);      // R is at most 128
  const int32_t g = threadIdx.x / per, c = 2 * (threadIdx.x - g * per);
  const int32_t tile = (int32_t)block * G + g;
  const bool cut = LONG && f.done != nullptr, two = c + 1 < f.R;
  const int32_t short_run = run_short(f.R, G);
  bool is_long = false, is_piece = false;        // is_piece: this tile's sum is a part of a cut run
  if (g < G && tile < f.num_tiles) {
    const int32_t seg_before = tile > 0 ? __ldg(f.carry_seg + tile - 1) : -2;
    const int32_t seg = __ldg(f.carry_seg + tile);
    const bool head = seg >= 0 && seg_before != seg;
    if (head || (seg >= 0 && cut && tile % kRunPiece == 0 && run_cut_at(f, tile, seg))) {
      const int32_t edge = (tile / kRunPiece + 1) * kRunPiece;
      const bool on = cut && run_cut_at(f, edge, seg);                     // the run goes on in a piece of its own
      const int32_t limit = on ? edge : f.num_tiles;                       // it is followed up to here
      auto carry = [&](int32_t t) {
        const double *at = f.carry_val + (int64_t)t * f.carry_ld + c;
        return f.carry_ld == 1 ? make_double2(__ldcs(at), 0.0) : __ldcs(reinterpret_cast<const double2 *>(at));
      };
      double2 sum = make_double2(0.0, 0.0);
      bool more = true;
      int32_t q = 0;
      for (int step = run_first(f.R); more && (!LONG || q < short_run); q += step, step = 8) {
        int32_t s[8];
        double2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const bool in = u < step && tile + q + u < limit;
          s[u] = in ? __ldg(f.carry_seg + tile + q + u) : -2;
          v[u] = in ? carry(tile + q + u) : make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (u < step) {
            more = more && s[u] == seg;
            if (more) { sum.x += v[u].x; sum.y += v[u].y; }
          }
        }
      }
      is_long = LONG && more;                    // every thread of the tile sees the same run
      if (!is_long) {
        if (head && !on) {
          const int64_t row = f.out_row ? (int64_t)__ldg(f.out_row + seg) : (int64_t)seg;
          T *const dst = static_cast<T *>(f.C) + row * f.ldc + c;
          const double x = (double)dst[0], y = two ? (double)dst[1] : 0.0;
          dst[0] = (T)(x + sum.x);
          if (two) dst[1] = (T)(y + sum.y);
        } else {
          f.carry_val[(int64_t)tile * f.carry_ld + c] = sum.x;
          if (two) f.carry_val[(int64_t)tile * f.carry_ld + c + 1] = sum.y;
        }
        is_piece = !head || on;
      }
    }
  }
  if constexpr (LONG) {
    if (!__syncthreads_or(is_long || is_piece)) return;
    __shared__ double s_part[kBlockThreads];
    __shared__ int32_t s_long[kBlockThreads], s_longs, s_old;
    if (threadIdx.x == 0) s_longs = 0;
    __syncthreads();
    if ((is_long || is_piece) && c == 0) s_long[atomicAdd(&s_longs, 1)] = is_long ? tile : ~tile;
    __syncthreads();
    const int32_t longs = s_longs;
    for (int32_t x = 0; x < longs; ++x) {
      const int32_t first = s_long[x] < 0 ? ~s_long[x] : s_long[x];
      const int32_t seg = __ldg(f.carry_seg + first);
      if (cut && s_long[x] < 0) {
        finish_piece<T>(f, first, seg, s_part, &s_old);
        continue;
      }
      const int32_t edge = (first / kRunPiece + 1) * kRunPiece;
      const bool on = cut && run_cut_at(f, edge, seg);
      const int32_t limit = on ? edge : f.num_tiles;
      int32_t count = short_run, more;
      do {
        const int32_t at = first + count + threadIdx.x;
        more = __syncthreads_count(at < limit && __ldg(f.carry_seg + at) == seg);
        count += more;
      } while (more == kBlockThreads);
      const double sum = cta_slot_sum(f, first, 1, count, s_part);
      if (threadIdx.x < f.R) {
        const bool head = first == 0 || __ldg(f.carry_seg + first - 1) != seg;
        if (head && !on) add_to_row<T>(f, seg, threadIdx.x, sum);
        else f.carry_val[(int64_t)first * f.carry_ld + threadIdx.x] = sum;
        if (threadIdx.x == 0) s_old = head && !on;
      }
      __syncthreads();
      if (cut && !s_old) finish_piece<T>(f, first, seg, s_part, &s_old);
      __syncthreads();
    }
  }
}

// ONE: a vector result (R = 1, slots without gaps, runs not cut), known to the compiler: the launch of some hundred CTAs is
// short enough that fetching its instructions shows (power-law matrix of 19.5 M entries times a vector 107.7 -> 105.6 us).
template <class T, bool ONE>
__global__ void __launch_bounds__(kBlockThreads) carry_fixup_kernel(FixupArgs f) {
  if (ONE) {
    f.R = 1;
    f.carry_ld = 1;
    f.ldc = 1;
    f.done = nullptr;
  }
  carry_fixup_role<T, true>(f, blockIdx.x);
}

static int64_t fixup_blocks(int64_t num_tiles, int32_t R) { return ceil_div(num_tiles, fixup_tiles(R)); }

// SpMM with the long-row path: both fix-ups in one launch. They read different scratch and write different rows
// of C (the general tiles leave the long rows out, so no carry names one), so the first `heavy_blocks` CTAs add
// the long rows' slots while the others add the carries. (Runs are short here: the general tiles' segments are shorter
// than the long-row threshold.)
template <class T>
__global__ void __launch_bounds__(kBlockThreads) spmm_fixups_kernel(const HeavyArgs h, int heavy_blocks, const FixupArgs f) {
  if ((int)blockIdx.x < heavy_blocks) heavy_fixup_role<T>(h, (int)blockIdx.x, heavy_blocks);
  else carry_fixup_role<T, false>(f, (int64_t)blockIdx.x - heavy_blocks);
}

int64_t carry_seg_words(int64_t num_tiles) { return num_tiles + num_tiles / kRunPiece + 2; }

void carry_fixup_launch(int dtype, double *carry_val, int32_t *carry_seg, int64_t num_tiles, int32_t R, int32_t carry_ld,
                        void *C, int64_t ldc, const int32_t *out_row, bool cut_runs, cudaStream_t stream) {
  const bool cut = cut_runs && num_tiles > 2 * kRunPiece;
  const FixupArgs f{carry_val, carry_seg, (int32_t)num_tiles, R, carry_ld, C, ldc, out_row, cut ? carry_seg + num_tiles : nullptr};
  const unsigned blocks = (unsigned)fixup_blocks(num_tiles, R);
  const bool one = R == 1 && carry_ld == 1 && ldc == 1 && !cut;
  if (dtype == COMET_F32) (one ? carry_fixup_kernel<float, true> : carry_fixup_kernel<float, false>)<<<blocks, kBlockThreads, 0, stream>>>(f);
  else (one ? carry_fixup_kernel<double, true> : carry_fixup_kernel<double, false>)<<<blocks, kBlockThreads, 0, stream>>>(f);
}

// Clears `rows` rows of `width` pieces (V: an element or 16 bytes), `ld` pieces apart, in one stream of stores: a CTA takes
// 2,048 consecutive pieces of the result, a division per thread finds the first and the steps between its eight are added.
template <class V>
__global__ void __launch_bounds__(256) zero_rows_kernel(V *__restrict__ C, int64_t rows, int64_t width, int64_t ld, int32_t step_rows,
                                                        int32_t step_cols) {
  const int64_t i0 = (int64_t)blockIdx.x * 2048 + threadIdx.x;
  int64_t r = i0 < (1ll << 32) && width < (1ll << 32) ? (int64_t)((uint32_t)i0 / (uint32_t)width) : i0 / width;
  int64_t c = i0 - r * width;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    if (r < rows) {
      if (ld == width) __stcs(C + c, V{});                 // one long row
      else C[r * ld + c] = V{};                            // the rest of a sector at a row's end may still come
    }
    r += step_rows;
    c += step_cols;
    if (c >= width) { c -= width; ++r; }
  }
}

comet_status_t zero_rows(Context *ctx, void *C, int dtype, int64_t rows, int64_t R, int64_t ldc, cudaStream_t stream) {
  if (rows <= 0 || R <= 0) return COMET_OK;
  if (ldc == R || rows == 1) { R *= rows; ldc = R; rows = 1; }             // no gaps: one long row
  const int64_t per = dtype == COMET_F32 ? 4 : 2;
  const bool wide = R % per == 0 && ldc % per == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
  const int64_t width = wide ? R / per : R, ld = wide ? ldc / per : ldc;
  const unsigned blocks = (unsigned)ceil_div(rows * width, 2048);
  const int32_t step_rows = (int32_t)(256 / width), step_cols = (int32_t)(256 % width);
  if (wide) zero_rows_kernel<int4><<<blocks, 256, 0, stream>>>((int4 *)C, rows, width, ld, step_rows, step_cols);
  else if (dtype == COMET_F32) zero_rows_kernel<float><<<blocks, 256, 0, stream>>>((float *)C, rows, width, ld, step_rows, step_cols);
  else zero_rows_kernel<double><<<blocks, 256, 0, stream>>>((double *)C, rows, width, ld, step_rows, step_cols);
  COMET_LAUNCH_CHECK(ctx);
  return COMET_OK;
}

static int32_t forced_tile_items() {
  if (const char *e = getenv("COMET_TILE_ITEMS")) {
    int v = atoi(e);
    if (v >= 8 && v <= (1 << 20)) return v;
  }
  return 0;
}

// Items per tile where tiles cost the same: one tile per resident worker (148 SMs x ctas_per_sm CTAs), so that the launch is one
// full wave, or, beyond `once` items, full waves, `waves` or more, of tiles of at most `most`. Every tile costs a boundary, a cold
// start and a carry, and a wave that is partly filled costs a whole one. With about 4 tiles per worker, rounded to at most 160 items
// on mid-sized inputs, -> as here: SpMM, fp64, 3.1 M entries, R = 32 99.7 -> 79.0 us, 5.6 M, R = 10 116.7 -> 106.6, 5 M, R = 64 350
// -> 322; TTM, R = 16, 3 M 74.3 -> 57.7, R = 32, 10 M 224 -> 196; MTTKRP, CSF, 3 M, R = 16 124 -> 107.5, COO, 20 M, R = 32 629 -> 592;
// two waves 88 / 114 / 335, 60.6 / 205, 114.
// Small inputs, whose full wave would be of tiles below `brief` items, take `few` CTAs per SM, mid-sized ones three of four: fewer
// and longer tiles, but whole CTAs per SM, or some SMs have one more than the others (COO MTTKRP, 1 M entries, fp64, R = 8 28.4 us
// with two, 35.0 with 2.2). SpMM of every width class, uniform and power-law rows, time over that of two CTAs per SM: full-wave
// tiles of 10 to 16 items 1.00 with three and 1.05 with four; 20 to 30 0.96 and 1.01; 45 to 60 0.95 and 0.95; 76 0.91 and 0.92.
int32_t choose_tile_items(int64_t total_items, int workers_per_block, int ctas_per_sm, const TileRule &r) {
  if (const int32_t forced = forced_tile_items()) return forced;
  auto with_ctas = [&](int64_t ctas) { return ceil_div(total_items, kSmCount * ctas * workers_per_block); };
  int64_t t = with_ctas(ctas_per_sm);
  if (t > r.once) t = with_ctas(ctas_per_sm * (ceil_div(t, r.most) > r.waves ? ceil_div(t, r.most) : r.waves));
  else if (t < r.brief) t = with_ctas(r.few);
  else if (ctas_per_sm == 4 && t < (workers_per_block < 64 ? 64 : 32)) t = with_ctas(3);
  return (int32_t)(t < r.least ? r.least : t);
}

// The same where tiles are uneven: beside the long rows of an SpMM, whose entries the tiles leave out, and where the rows of a
// cleared C are written far apart. Four tiles per resident worker, or eight, so that the last ones do not leave the
// chip idle. DCSR, 94 % of the rows empty, R = 8, 2 / 4 / 6 / 8 tiles 1037 / 960 / 928 / 919 us; 5.6 M entries in power-law rows,
// R = 32, one / two / four / eight 478 / 456 / 454 / 422 us; 4.2 M rows in a cleared C, R = 8, one wave 788, eight tiles 762.
// Not that many where the tiles would be below `low` items, while half of the workers have one: beside long rows 160 (1.4 M entries in
// equal rows, fp32, R = 64 95 us with at least 32, 80 with 160; power-law rows, fp64, R = 128 184 and 180), in a cleared C 32.
static int32_t choose_uneven_tile_items(int64_t total_items, int workers_per_block, int per_worker, int32_t low) {
  if (const int32_t forced = forced_tile_items()) return forced;
  const int64_t slots = (int64_t)kSmCount * 4 * workers_per_block;
  int64_t t = ceil_div(total_items, slots * per_worker);
  const int64_t half = ceil_div(total_items, (int64_t)kSmCount * 2 * workers_per_block);
  const int64_t least = half < 8 ? 8 : half < low ? half : low;
  if (t < least) t = least;
  return (int32_t)(t < 512 ? t : 512);
}

template <class T, int LPN, int CPL, int VEC, bool RAGGED, int ROWS, bool HEAVY>
static comet_status_t launch_mapped(Context *ctx, const SegGatherArgs &a, const HeavyArgs &h, int64_t blocks,
                                    cudaStream_t stream) {
  using L = Lanes<T, LPN, CPL, VEC, RAGGED>;
  constexpr size_t ring = RingLayout<L, false>::kBlockBytes, async_ring = HEAVY ? AsyncRing<L>::kBlockBytes : 0;
  constexpr size_t smem = ring > async_ring ? ring : async_ring;
  static_assert(ROWS != kRowsMapped || smem >= kGapRows / 8 + 4 + kGapRows * 2, "gap_role: marks, their number, the empty rows");
  auto kernel = seg_gather_kernel<T, LPN, CPL, VEC, RAGGED, ROWS, HEAVY>;
  if (smem > 48 * 1024)
    COMET_CUDA_TRY(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  kernel<<<(unsigned)(blocks + (HEAVY ? h.heavy_ctas : 0)), kBlockThreads, smem, stream>>>(a, h);
  COMET_LAUNCH_CHECK(ctx);
  return COMET_OK;
}

// The shapes whose rows are 256, 512 or 1024 bytes carry the long-row role of SpMM.
template <class T, int LPN, int CPL, int VEC> constexpr bool kHeavyShape =
    VEC * sizeof(T) == 16 && (LPN * CPL * VEC * sizeof(T) == 256 || LPN * CPL * VEC * sizeof(T) == 512 ||
                              LPN * CPL * VEC * sizeof(T) == 1024) && LPN >= 16;

static size_t carry_bytes(int64_t num_tiles, int32_t carry_ld) {
  return align_up((size_t)num_tiles * carry_ld * sizeof(double), 256) + align_up((size_t)carry_seg_words(num_tiles) * sizeof(int32_t), 256);
}

// What has to be there before a gather kernel starts, as roles of one launch (the steps are latency, not data: side by side
// they cost what the longest of them does): copies of dense rows padded with zeros to whole 16-byte pieces, a thread per
// piece, and in front of them, for SpMM and TTM, the merge-path split at every tile boundary, a thread per boundary.
struct PadJob {
  const void *src;
  int64_t pieces_total;      // rows * pieces
  int64_t ld;
  void *dst;
  int32_t R, pieces;
};
struct PrepareArgs {
  const int32_t *seg_end;
  int64_t M, N, num_tiles;
  int32_t tile_items;
  int32_t *part;
  int64_t part_blocks;
  PadJob pad[2];
  int64_t pad_blocks[2];
};

template <class T>
__device__ __forceinline__ void pad_role(const PadJob &p, int64_t i) {
  constexpr int PER = 16 / sizeof(T);
  if (i >= p.pieces_total) return;
  const int64_t r = i < (1ll << 31) ? (int64_t)((uint32_t)i / (uint32_t)p.pieces) : i / p.pieces;
  const int32_t c = (int32_t)(i - r * p.pieces) * PER;
  const T *src = static_cast<const T *>(p.src) + r * p.ld + c;
  T v[PER];
#pragma unroll
  for (int x = 0; x < PER; ++x) v[x] = c + x < p.R ? __ldg(src + x) : (T)0;
  reinterpret_cast<int4 *>(p.dst)[i] = *reinterpret_cast<const int4 *>(v);
}

template <class T>
__global__ void __launch_bounds__(kBlockThreads) prepare_kernel(const PrepareArgs a) {
  int64_t block = blockIdx.x;
  if (block < a.part_blocks) {
    const int64_t t = block * kBlockThreads + threadIdx.x;
    if (t > a.num_tiles) return;
    const int64_t total = a.M + a.N;
    const int64_t d = t * a.tile_items < total ? t * a.tile_items : total;
    a.part[t] = (int32_t)merge_path_segments(a.seg_end, a.M, a.N, d);
    return;
  }
  block -= a.part_blocks;
  if (block < a.pad_blocks[0]) { pad_role<T>(a.pad[0], block * kBlockThreads + threadIdx.x); return; }
  pad_role<T>(a.pad[1], (block - a.pad_blocks[0]) * kBlockThreads + threadIdx.x);
}

size_t padded_bytes(int dtype, int64_t rows, int64_t R) {
  const int per = dtype == COMET_F32 ? 4 : 2;
  return align_up((size_t)rows * ceil_div(R, per) * 16, 256);
}
static void pad_job(PrepareArgs &a, int which, int dtype, const void *src, int64_t rows, int64_t R, int64_t ld, void *dst) {
  PadJob &p = a.pad[which];
  p.src = src; p.ld = ld; p.dst = dst; p.R = (int32_t)R;
  p.pieces = (int32_t)ceil_div(R, dtype == COMET_F32 ? 4 : 2);
  p.pieces_total = rows * p.pieces;
  a.pad_blocks[which] = ceil_div(p.pieces_total, (int64_t)kBlockThreads);
}
static comet_status_t prepare_run(Context *ctx, int dtype, const PrepareArgs &a, cudaStream_t stream) {
  const int64_t blocks = a.part_blocks + a.pad_blocks[0] + a.pad_blocks[1];
  if (blocks == 0) return COMET_OK;
  if (dtype == COMET_F32) prepare_kernel<float><<<(unsigned)blocks, kBlockThreads, 0, stream>>>(a);
  else prepare_kernel<double><<<(unsigned)blocks, kBlockThreads, 0, stream>>>(a);
  COMET_LAUNCH_CHECK(ctx);
  return COMET_OK;
}
comet_status_t pad_rows2(Context *ctx, int dtype, const void *src0, int64_t rows0, int64_t ld0, void *dst0, const void *src1, int64_t rows1,
                         int64_t ld1, void *dst1, int64_t R, cudaStream_t stream) {
  PrepareArgs a{};
  pad_job(a, 0, dtype, src0, rows0, R, ld0, dst0);
  pad_job(a, 1, dtype, src1, rows1, R, ld1, dst1);
  return prepare_run(ctx, dtype, a, stream);
}

// A worker of one lane reads its tile's entries by itself, 32 such tiles to a warp: where they are long, no two lanes read from
// one line, and all the lines are more than the L1 holds. 12 to 18 entries are best at every size: SpMM of 9 M entries, fp64, R = 2
// 522 us in one wave, 517 with four tiles per worker, 228 as here; fp32, R = 4 452, 453 and 183; TTM, fp64 518, 368 and 224. Two lanes and more: 1,024 entries are added in a row at most.
// Where a tensor's fibers are long on average (`mixed`), some tiles may hold nothing but short ones, which store a row per entry or
// two, and in one wave the launch waits for those: three waves from 192 items on (16 lanes: 400), for the workers that do not fill a warp. Slices
// of very different sizes, 22 entries per fiber, 9 M, fp64, R = 10 135 us with four tiles per worker, 162 in one wave, 146 as here; fp32,
// R = 50, 5.5 M 186, 210 and 173. With short fibers everywhere tiles are alike (8 per fiber, 3.2 M, fp64, R = 32 95 us with four tiles
// per worker, 74 in one wave, 92 in three); in matrices the long rows cost what the short ones do.
template <int LPN>
constexpr TileRule gather_tile_rule(bool mixed) {
  if (LPN == 1) return TileRule{8, 12, 2, 20, 1, 16};
  return mixed && LPN < 32 ? TileRule{8, 24, 2, LPN == 16 ? 400 : 192, 3, 640} : TileRule{8, 24, 2, 1024, 1, 1024};
}

// `heavy` (optional): the long-row plan of an SpMM; its scratch precedes the carries of this launch. pad (RAGGED): the
// first `pad` rows of B are copied into scratch as whole pieces and gathered from there. cleared: out_row is given and C
// holds zeros. fibers: segments are fibers of a tensor.
template <class T, int LPN, int CPL, int VEC, bool RAGGED = false>
static comet_status_t launch_one(Context *ctx, SegGatherArgs a, HeavyArgs *heavy, bool cleared, bool fibers, int64_t pad, cudaStream_t stream, int32_t at_least = 0) {
  constexpr int WORKERS = kBlockThreads / LPN;
  const int64_t total = a.M + a.N;
  a.carry_ld = (int32_t)align_up((size_t)a.R, 2);
  constexpr int kCtas = resident_ctas(CPL * VEC * sizeof(T) <= 16 ? COMET_MINB_GATHER : 2, RingLayout<Lanes<T, LPN, CPL, VEC, RAGGED>, false>::kBlockBytes);
  TileRule rule = gather_tile_rule<LPN>(fibers && a.N >= 12 * a.M);
  if (a.out_row && !cleared && kCtas == 2) { rule.brief = 96; rule.few = 1; }           // the CTAs that clear rows run beside them
  a.tile_items = a.out_row && cleared && LPN > 1 ? choose_uneven_tile_items(total, WORKERS, 8, 32) : choose_tile_items(total, WORKERS, kCtas, rule);
  // a bound on the carries, which the handle's scratch keeps (up to 40 bytes per tile): four million short tiles
  if (LPN == 1 && at_least < total >> 22) at_least = (int32_t)(total >> 22);
  if (a.tile_items < at_least) a.tile_items = at_least;
  size_t heavy_bytes = 0;
  HeavyArgs h{};
  if (!RAGGED && kHeavyShape<T, LPN, CPL, VEC> && heavy && !a.out_row) {
    const int32_t tile = choose_uneven_tile_items(total, WORKERS, 4, 160);
    heavy_bytes = spmm_heavy_plan(sizeof(T) == 4 ? COMET_F32 : COMET_F64, a.M, a.N, heavy->cols, a.B, a.ldb, a.R, a.C, a.ldc, tile, &h);
    if (heavy_bytes) a.tile_items = tile;
  }
  a.num_tiles = ceil_div(total, a.tile_items);
  a.own_len = a.tile_items / 4;
  const size_t val_bytes = align_up((size_t)a.num_tiles * a.carry_ld * sizeof(double), 256);
  static const bool use_part = !(getenv("COMET_SEG_PARTITION") && atoi(getenv("COMET_SEG_PARTITION")) == 0);
  constexpr int kDtype = sizeof(T) == 4 ? COMET_F32 : COMET_F64;
  const size_t pad_bytes = RAGGED && pad ? padded_bytes(kDtype, pad, a.R) : 0;
  // The split at the tile boundaries as a launch of its own costs 3 us; a worker that finds its own boundaries takes
  // log2(M) / log2(LPN) dependent loads. So it pays from about a thousand tiles with few lanes (or beside padded copies or
  // the long-row plan, which need the launch anyway), from many thousands with more: with the launch from 1,024 tiles at every
  // width, SpMM of 89,000 entries in 16-lane workers took 21.7 us instead of 12.5, of 45,000 in whole warps 16.6 instead of
  // 13.9; from 16,384 tiles on both are the same. In 2-lane workers the launch takes 25,000 entries from 22 to 13 us.
  const int64_t part_least = LPN <= 4 || pad_bytes || heavy_bytes ? 1024 : 16384;
  const size_t part_bytes = use_part && a.num_tiles >= part_least ? align_up((size_t)(a.num_tiles + 1) * sizeof(int32_t), 256) : 0;
  char *scratch = (char *)scratch_get(ctx, pad_bytes + heavy_bytes + carry_bytes(a.num_tiles, a.carry_ld) + part_bytes, stream);
  // many short tiles have many carries: with no room for them, longer tiles
  if (!scratch && LPN == 1 && a.tile_items < 512) return launch_one<T, LPN, CPL, VEC, RAGGED>(ctx, a, heavy, cleared, fibers, pad, stream, 512);
  if (!scratch) return COMET_ERR_ALLOC;
  PrepareArgs prep{};
  if (pad_bytes) {
    pad_job(prep, 0, kDtype, a.B, pad, a.R, a.ldb, scratch);
    a.B = scratch;
    a.ldb = ceil_div(a.R, VEC) * VEC;
    scratch += pad_bytes;
  }
  a.carry_val = (double *)(scratch + heavy_bytes);
  a.carry_seg = (int32_t *)(scratch + heavy_bytes + val_bytes);
  if (part_bytes) {
    int32_t *part = (int32_t *)(scratch + heavy_bytes + carry_bytes(a.num_tiles, a.carry_ld));
    if (heavy_bytes) {                                     // a role of the long-row path's pieces launch
      h.part_seg_end = a.seg_end; h.part_M = a.M; h.part_N = a.N; h.part_tiles = a.num_tiles;
      h.part_tile_items = a.tile_items; h.part = part;
    } else {
      prep.seg_end = a.seg_end; prep.M = a.M; prep.N = a.N; prep.num_tiles = a.num_tiles;
      prep.tile_items = a.tile_items; prep.part = part;
      prep.part_blocks = ceil_div(a.num_tiles + 1, (int64_t)kBlockThreads);
    }
    a.part = part;
  }
  const int64_t blocks = ceil_div(a.num_tiles, WORKERS);
  comet_status_t st = prepare_run(ctx, kDtype, prep, stream);
  if (st != COMET_OK) return st;
  if constexpr (!RAGGED && kHeavyShape<T, LPN, CPL, VEC>) {
    if (heavy_bytes) {
      st = spmm_heavy_prepare(ctx, &h, a.seg_end - 1, a.crd, a.val, scratch, stream);
      if (st != COMET_OK) return st;
      a.skip_len = h.threshold;
      st = launch_mapped<T, LPN, CPL, VEC, false, kRowsAll, true>(ctx, a, h, blocks, stream);
      if (st != COMET_OK) return st;
      const int heavy_blocks = kSmCount * 8;
      const unsigned fix_blocks = (unsigned)(heavy_blocks + fixup_blocks(a.num_tiles, a.R));
      const FixupArgs f{a.carry_val, a.carry_seg, (int32_t)a.num_tiles, a.R, a.carry_ld, a.C, a.ldc, nullptr, nullptr};
      spmm_fixups_kernel<T><<<fix_blocks, kBlockThreads, 0, stream>>>(h, heavy_blocks, f);
      COMET_LAUNCH_CHECK(ctx);
      return COMET_OK;
    }
  }
  a.gap_from = blocks;
  const int64_t gap_blocks = a.out_row && !cleared ? ceil_div(a.out_rows, (int64_t)kGapRows) : 0;
  st = !a.out_row ? launch_mapped<T, LPN, CPL, VEC, RAGGED, kRowsAll, false>(ctx, a, h, blocks, stream)
                  : launch_mapped<T, LPN, CPL, VEC, RAGGED, kRowsMapped, false>(ctx, a, h, blocks + gap_blocks, stream);
  if (st != COMET_OK) return st;
  carry_fixup_launch(kDtype, a.carry_val, a.carry_seg, a.num_tiles, a.R, a.carry_ld, a.C, a.ldc, a.out_row, true, stream);
  COMET_LAUNCH_CHECK(ctx);
  return COMET_OK;
}

static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// One launch per chunk of up to 128 columns. A power-of-two number of whole pieces on aligned rows takes an exact
// shape, anything else a ragged one; rows of B that are no whole pieces are padded into scratch first, unless B has so
// many more rows than the matrix has entries that the copy would cost more than it saves: then the scalar shapes (32
// lanes, a column each) run on B as it is. What the scalar shapes lose is lanes (R = 10: 22 of 32 idle) and requests in
// flight. Measured, scalar -> ragged: 4 M entries in 200,000 rows, R = 3 / 10 / 25 / 50 / 100 fp64 134 -> 68, 137 -> 77, 155
// -> 122, 194 -> 167, 463 -> 403 us, fp32 129 -> 70, 132 -> 77, 136 -> 109, 187 -> 151, 304 -> 208 us; a power-law
// matrix of 3.2 M entries, R = 50, fp32 156 -> 145 us. Small inputs have the scalar shapes too, unless the ragged one is a
// whole warp that reads B as it is: many narrow workers to a CTA leave few CTAs, and each finds its tile with few lanes. Over
// some thousand random inputs the two are level between 150,000 (up to 4 lanes) and 500,000 entries (16 lanes, or copies);
// below, the ragged ones took up to 1.7 times as long (34,700 entries, fp64, R = 24 20.7 us, scalar 12.1; 97,000, R = 20 27.8,
// scalar 18.6).
constexpr int64_t kRaggedLeastNarrow = 150000, kRaggedLeast = 250000;      // up to four pieces, more

template <class T>
static comet_status_t seg_gather_typed(Context *ctx, const int32_t *seg_end, const int32_t *crd, const T *val,
                                       int64_t M, int64_t N, const T *B, int64_t ldb, int64_t R, T *C, int64_t ldc,
                                       const int32_t *out_row, int64_t out_rows, int64_t b_rows, bool long_rows,
                                       bool fibers, cudaStream_t stream) {
  constexpr int PER = 16 / sizeof(T);                      // elements per 128-bit piece
  HeavyArgs hint{};                                        // SpMM on [D,CU]: long rows by column phases
  hint.cols = b_rows;
  HeavyArgs *heavy = long_rows && !out_row && b_rows > 0 && R <= 128 ? &hint : nullptr;
  const bool b_ok = aligned16(B) && ldb % PER == 0, c_ok = aligned16(C) && ldc % PER == 0;
  // The copy moves a row of B twice (0.4 ps per byte and row); a ragged shape saves about 17 ps per entry on the scalar one.
  bool pad = N >= (R <= 4 * PER ? kRaggedLeastNarrow : kRaggedLeast) && N * 40 >= b_rows * R * (int64_t)sizeof(T);
  // More than 32 pieces are two per lane, which halves the warps on an SM. Long rows of a B that stays in L2 are faster as
  // two launches of at most 32 (4 M entries in 200,000 rows, 84 MB of B: R = 70 335 -> 262 us), short ones, a B in DRAM and
  // small inputs (35,000 entries: 22 -> 40 us) are not (2.9 entries per row: 784 -> 1128 us; 430 MB: 398 -> 527 us). Short
  // rows are faster still with a column per lane (R = 70: 784 -> 760 us): what costs there is the stores of the ragged rows;
  // and so is more than 96 columns where two launches would be of nearly the same width (DCSR, 1.6 M entries, R = 100 457 ->
  // 277 us; 2.1 M, R = 127 225 -> 189 us).
  const bool split = N >= (1 << 20) && N >= 8 * M && b_rows * R * (int64_t)sizeof(T) <= (126ll << 20);
  auto one_column_per_lane = [&](int64_t chunk) {
    return chunk > 32 * PER && ((chunk < 64 * PER && N < 4 * M) || (split && R <= 128 && chunk > 48 * PER));
  };
  // A compressed root level whose empty rows are cleared by CTAs of the gather launch (gap_role), which write them once, or
  // C is cleared as a whole in one stream of wide stores first (7.5 TB/s where the others reach 4.5) and the stored rows are written over
  // it: narrow rows, or few stored ones in a large C. Gaps -> stream: 4.2 M entries in 67 M / 8.4 M rows, R = 8 1018 -> 765, 269 ->
  // 232 us; 1 M in 5 M, fp32, R = 4 92 -> 65; 0.13 M in 0.76 M, R = 19 57 -> 46; 0.16 M in 1.6 M, fp32, R = 2 29 -> 23; 3.2 M in 7 M, R = 25 606
  // -> 530; 5.5 M in 7.3 M, fp32, R = 4 294 -> 227; but 1 M in 3 M, R = 64 331 -> 395; 0.32 M in 1.06 M, R = 25 82 -> 97; 42,000 in 282,000,
  // fp32, R = 32 the stream takes 1.4 times as long.
  const int64_t row_bytes = R * (int64_t)sizeof(T), c_bytes = out_rows * row_bytes;
  const bool cleared = out_row && (out_rows >= 6 * M ? c_bytes >= (row_bytes <= 64 ? 10000000 : 100000000)
                                   : out_rows >= 2 * M ? (row_bytes <= 64 && c_bytes >= 20000000) || (row_bytes <= 256 && c_bytes >= 1000000000)
                                                       : 2 * out_rows >= 3 * M && row_bytes <= 16 && c_bytes >= 50000000);
  if (cleared) {
    const comet_status_t zs = zero_rows(ctx, C, sizeof(T) == 4 ? COMET_F32 : COMET_F64, out_rows, R, ldc, stream);
    if (zs != COMET_OK) return zs;
  }
  int64_t done = 0;
  while (done < R) {
    SegGatherArgs a{};
    a.seg_end = seg_end; a.crd = crd; a.val = val; a.M = M; a.N = N;
    a.B = B + done; a.ldb = ldb; a.C = C + done; a.ldc = ldc;
    a.out_row = out_row; a.out_rows = out_rows;
    a.wide_store = c_ok;
    comet_status_t st = COMET_OK;
    const int64_t rem = R - done;
    int64_t chunk = rem < 128 ? rem : 128;
    const bool whole = b_ok && chunk % PER == 0;           // gathered from B as it is, in whole pieces
    const bool wide = whole && c_ok && chunk == 64 * PER;
    bool pieces_ok = (whole || pad) && (wide || !one_column_per_lane(chunk));
    if (pieces_ok && chunk > 32 * PER && split && !wide) chunk = 32 * PER;
    const int64_t pieces = ceil_div(chunk, PER);
    const bool exact = whole && c_ok && (pieces & (pieces - 1)) == 0;
    if (whole && !exact && pieces <= 16 && N < (pieces <= 4 ? kRaggedLeastNarrow : kRaggedLeast)) pieces_ok = false;
    a.R = (int32_t)chunk;
    if (pieces_ok) {
      const int64_t p = whole ? 0 : b_rows;
      if (pieces > 32) {
        if constexpr (sizeof(T) == 8)                      // fp32 chunks are at most 32 pieces
          st = exact ? launch_one<T, 32, 2, PER>(ctx, a, heavy, cleared, fibers, 0, stream) : launch_one<T, 32, 2, PER, true>(ctx, a, heavy, cleared, fibers, p, stream);
      } else if (exact && pieces == 32) st = launch_one<T, 32, 1, PER>(ctx, a, heavy, cleared, fibers, 0, stream);
      else if (exact && pieces == 16) st = launch_one<T, 16, 1, PER>(ctx, a, heavy, cleared, fibers, 0, stream);
      else if (exact && pieces == 8) st = launch_one<T, 8, 1, PER>(ctx, a, heavy, cleared, fibers, 0, stream);
      else if (exact && pieces == 4) st = launch_one<T, 4, 1, PER>(ctx, a, heavy, cleared, fibers, 0, stream);
      else if (exact && pieces == 2) st = launch_one<T, 2, 1, PER>(ctx, a, heavy, cleared, fibers, 0, stream);
      else if (exact && pieces == 1) st = launch_one<T, 1, 1, PER>(ctx, a, heavy, cleared, fibers, 0, stream);
      else if (pieces > 16) st = launch_one<T, 32, 1, PER, true>(ctx, a, heavy, cleared, fibers, p, stream);
      else if (pieces > 8) st = launch_one<T, 16, 1, PER, true>(ctx, a, heavy, cleared, fibers, p, stream);
      else if (pieces > 4) st = launch_one<T, 8, 1, PER, true>(ctx, a, heavy, cleared, fibers, p, stream);
      else if (pieces > 2) st = launch_one<T, 4, 1, PER, true>(ctx, a, heavy, cleared, fibers, p, stream);
      else st = launch_one<T, 2, 1, PER, true>(ctx, a, heavy, cleared, fibers, p, stream);
    } else {
      if (a.R > 64) st = launch_one<T, 32, 4, 1>(ctx, a, heavy, cleared, fibers, 0, stream);
      else if (a.R > 32) st = launch_one<T, 32, 2, 1>(ctx, a, heavy, cleared, fibers, 0, stream);
      else st = launch_one<T, 32, 1, 1>(ctx, a, heavy, cleared, fibers, 0, stream);
    }
    if (st == COMET_ERR_ALLOC && pieces_ok && !whole) {       // no room for a padded copy: the shapes that need none
      pad = false;
      continue;
    }
    if (st != COMET_OK) return st;
    done += a.R;
  }
  return COMET_OK;
}

comet_status_t seg_gather(Context *ctx, int dtype, const int32_t *seg_end, const int32_t *crd, const void *val,
                          int64_t M, int64_t N, const void *B, int64_t ldb, int64_t R, void *C, int64_t ldc,
                          const int32_t *out_row, int64_t out_rows, int64_t b_rows, bool long_rows, bool fibers, cudaStream_t stream) {
  if (ldb >= (1ll << 28)) return COMET_ERR_INDEX_OVERFLOW;      // row offsets are formed as int32 bytes * int32 index
  if (M == 0) return out_row ? zero_rows(ctx, C, dtype, out_rows, R, ldc, stream) : COMET_OK;
  if (out_row && M == out_rows) out_row = nullptr;         // every row is stored: segment s is row s
  if (dtype == COMET_F32)
    return seg_gather_typed<float>(ctx, seg_end, crd, (const float *)val, M, N, (const float *)B, ldb, R, (float *)C, ldc,
                                   out_row, out_rows, b_rows, long_rows, fibers, stream);
  return seg_gather_typed<double>(ctx, seg_end, crd, (const double *)val, M, N, (const double *)B, ldb, R, (double *)C,
                                  ldc, out_row, out_rows, b_rows, long_rows, fibers, stream);
}

}  // namespace comet

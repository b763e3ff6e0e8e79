// MTTKRP of a CSF tensor [CU,CU,CU] for the output mode stored at level 1 (the textbook matricised-tensor-times-Khatri-Rao
// product the paper names): per fiber (i, j) of entries (i, j, k), out[j, :] += (sum of x * Q[k, :]) * P[i, :]. The fibers
// of one output row are spread over the whole tensor, so the sums go out as atomic adds in double, one row add per fiber.
//
// A worker is a warp (a half warp up to 16 columns); lane g owns columns g, g + G: any width and alignment, and both the
// row reads and the atomic adds of a row are contiguous requests. A worker walks a tile of up to 1,024 consecutive entries in
// chunks of 32:
//   * where fibers and slices end is known as two bit masks per chunk, formed for the whole tile before the walk by one
//     coalesced sweep over the fiber ends that fall into it, so the walk tests bits of a register instead of following
//     positions;
//   * the entries are staged one chunk ahead into a shared-memory ring as (value, k, j) and read back by broadcast;
//   * the Q rows of the next kPF entries are in flight in a rolling register window.
//
// What bounds it: instruction issue (27 per entry and 32 columns, 55 to 60 % issued) and the L1 data pipe. Measured against
// the walker of the root modes (fp64) or one worker per eight fibers (fp32, odd widths), which this replaces: 100 M
// entries, R = 32, fp64 4.03 -> 3.61 ms; 3 M, R = 25, fp32 358 -> 168 us; 5 M, R = 33 / 100, fp64 811 -> 421 / 1447 -> 920 us.
// 2, 4 and 8 rows in flight: 4.14 / 3.61 / 3.59 ms; 3 CTAs per SM 3.72; half warps with two columns per lane 3.82.
#include <stdlib.h>

#include "common.cuh"
#include "kernels.cuh"
#include "walk.cuh"

namespace comet {

constexpr int kLevel1Cap = 1024;                 // entries per tile at most
constexpr int kLevel1Words = kLevel1Cap / 32;
constexpr int kLevel1RingBytes = 2 * 32 * 16;
constexpr int kLevel1WorkerBytes = kLevel1RingBytes + 3 * kLevel1Words * 4 + 16;   // the skew keeps half warps on different banks

struct Level1Args {
  const int32_t *pos1, *crd0, *crd1, *seg_end2, *crd2;   // S + 1, S, F, F (= pos2 + 1), N
  const void *val;
  int64_t S, F, N;
  const void *P, *Q;
  int64_t ldp, ldq;
  double *acc;
  int64_t ldacc;
  int32_t R;
  int32_t tile;                                  // entries per tile, a multiple of 32
  int64_t num_tiles;
  const int32_t *part_fiber, *part_slice;        // per tile boundary
};

// First fiber that ends behind each tile boundary and the slice that holds it, a thread per boundary.
__global__ void __launch_bounds__(kBlockThreads) level1_starts_kernel(const int32_t *__restrict__ seg_end2,
                                                                      const int32_t *__restrict__ pos1, int64_t S, int64_t F,
                                                                      int64_t N, int32_t tile, int64_t num_tiles,
                                                                      int32_t *__restrict__ part_fiber,
                                                                      int32_t *__restrict__ part_slice) {
  const int64_t t = (int64_t)blockIdx.x * kBlockThreads + threadIdx.x;
  if (t > num_tiles) return;
  const int64_t j = t * tile < N ? t * tile : N;
  int64_t lo = 0, hi = F;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int64_t)__ldg(seg_end2 + mid) <= j) lo = mid + 1; else hi = mid;
  }
  const int64_t f = lo;
  part_fiber[t] = (int32_t)f;
  lo = 0, hi = S;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int64_t)__ldg(pos1 + mid + 1) <= f) lo = mid + 1; else hi = mid;
  }
  part_slice[t] = (int32_t)lo;
}

__device__ __forceinline__ void red_or_shared(uint32_t addr, uint32_t bits) {
  asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(addr), "r"(bits) : "memory");
}

// if (bit) { *p += t * r (atomic); t = 0; } Predicated, not branched: whether a fiber ends at an entry is a coin toss, and
// a branch per entry with its reconvergence costs more (50 instructions per entry instead of 27).
__device__ __forceinline__ void add_if(uint32_t bit, double *p, double &t, double r) {
  asm volatile("{.reg .pred p; .reg .f64 x; setp.ne.u32 p, %2, 0; mul.rn.f64 x, %0, %3; @p red.global.add.f64 [%1], x; "
               "@p mov.f64 %0, 0d0000000000000000;}"
               : "+d"(t) : "l"(p), "r"(bit), "d"(r) : "memory");
}

template <class T, int G, int CPL>
__global__ void __launch_bounds__(kBlockThreads, 4) mttkrp_level1_kernel(const Level1Args a) {
  constexpr int kPer = 32 / G;                   // entries a lane stages per chunk
  constexpr int kPF = 4;                         // Q rows in flight
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int worker = threadIdx.x / G, g = threadIdx.x & (G - 1);
  const int64_t tile = (int64_t)blockIdx.x * (kBlockThreads / G) + worker;
  if (tile >= a.num_tiles) return;               // whole groups leave together
  const int shift = threadIdx.x & 31 & ~(G - 1);
  const unsigned mask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << shift;
  const uint32_t ring = smem_u32(smem_raw) + worker * kLevel1WorkerBytes;
  const uint32_t w_ends = ring + kLevel1RingBytes, w_slices = w_ends + kLevel1Words * 4, w_rank = w_slices + kLevel1Words * 4;

  // Entries are counted from the tile's first one: the staging looks up to 96 entries ahead, and a tensor may hold so many
  // that their numbers do not fit 32 bits there.
  const int64_t first = tile * a.tile;
  const int32_t j0 = (int32_t)first, len = (int32_t)(a.N - first < a.tile ? a.N - first : a.tile);
  const T *const val = static_cast<const T *>(a.val) + first;
  const int32_t *const crd2 = a.crd2 + first;
  int32_t col[CPL];                              // a lane beyond the last column reads the last one and adds nothing
  bool ok[CPL];
#pragma unroll
  for (int t = 0; t < CPL; ++t) {
    ok[t] = g + t * G < a.R;
    col[t] = ok[t] ? g + t * G : a.R - 1;
  }
  const char *const qcol = reinterpret_cast<const char *>(static_cast<const T *>(a.Q) + col[0]);
  const char *const pcol = reinterpret_cast<const char *>(static_cast<const T *>(a.P) + col[0]);
  const uint32_t ldq_bytes = (uint32_t)(a.ldq * sizeof(T)), ldp_bytes = (uint32_t)(a.ldp * sizeof(T));
  auto gather = [&](const char *base, uint32_t ld_bytes, int32_t c, T (&dst)[CPL][1]) {
    const T *row = reinterpret_cast<const T *>(base + (uint64_t)(uint32_t)c * ld_bytes);
#pragma unroll
    for (int t = 0; t < CPL; ++t) Piece<T, 1>::load(t == 0 ? row : row + (col[t] - col[0]), dst[t]);
  };

  // ---- the masks of the tile. A caller's tensor may hold fibers or slices without entries: their ends fall on the bit of
  // the one in front, the bits are then fewer than the fibers (slices), and these are found by position instead.
  bool odd_fibers, odd_slices;
  const int32_t f0 = __ldg(a.part_fiber + tile), f1 = __ldg(a.part_fiber + tile + 1);     // fibers f0 .. f1-1 end in the tile
  int32_t s = __ldg(a.part_slice + tile);
  {
    const int32_t s1 = __ldg(a.part_slice + tile + 1);
    for (int w = g; w < 2 * kLevel1Words; w += G) sts_s32(w_ends + w * 4, 0);
    __syncwarp(mask);
    for (int32_t k = f0 + g; k < f1; k += 4 * G) {
      int32_t e[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) e[u] = k + u * G < f1 ? __ldg(a.seg_end2 + k + u * G) : 0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int32_t q = e[u] - 1 - j0;
        if (k + u * G < f1) red_or_shared(w_ends + (q >> 5) * 4, 1u << (q & 31));
      }
    }
    for (int32_t k = s + g; k < s1; k += G) {    // slice k ends with fiber pos1[k + 1] - 1
      const int32_t q = __ldg(a.seg_end2 + __ldg(a.pos1 + k + 1) - 1) - 1 - j0;
      red_or_shared(w_slices + (q >> 5) * 4, 1u << (q & 31));
    }
    __syncwarp(mask);
    constexpr int kOwn = kLevel1Words / G;       // words per lane
    int32_t cnt[kOwn], mine = 0, closed = 0;     // fiber ends in front of each word
#pragma unroll
    for (int i = 0; i < kOwn; ++i) {
      cnt[i] = mine;
      mine += __popc((uint32_t)lds_s32(w_ends + (g * kOwn + i) * 4));
      closed += __popc((uint32_t)lds_s32(w_slices + (g * kOwn + i) * 4));
    }
#pragma unroll
    for (int d = 1; d < G; d <<= 1) closed += __shfl_xor_sync(mask, closed, d, G);
    odd_slices = closed != s1 - s;
    int32_t inc = mine;
#pragma unroll
    for (int d = 1; d < G; d <<= 1) {
      const int32_t x = __shfl_up_sync(mask, inc, d, G);
      if (g >= d) inc += x;
    }
#pragma unroll
    for (int i = 0; i < kOwn; ++i) sts_s32(w_rank + (g * kOwn + i) * 4, inc - mine + cnt[i]);
    __syncwarp(mask);
    odd_fibers = __shfl_sync(mask, inc, G - 1, G) != f1 - f0;
  }
  auto fiber_of_end = [&](int32_t j) {           // the fiber whose last entry is the tile's entry j
    int32_t lo = f0, hi = f1;
    while (lo < hi) {
      const int32_t mid = lo + ((hi - lo) >> 1);
      if (__ldg(a.seg_end2 + mid) - j0 <= j) lo = mid + 1; else hi = mid;
    }
    return lo;
  };
  auto next_slice = [&](int32_t j) {             // the slice of the entry behind the tile's entry j
    ++s;
    if (odd_slices)
      while (s < a.S && __ldg(a.seg_end2 + __ldg(a.pos1 + s + 1) - 1) - j0 <= j + 1) ++s;
    return s < a.S;
  };

  // ---- staging
  double sv[kPer];
  int32_t sk[kPer], sj[kPer];
  auto load = [&](int32_t base) {                // base may run past the tile: idle entries
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int x = g + i * G;
      const int32_t j = base + x;
      sv[i] = 0.0;
      sk[i] = sj[i] = 0;
      if (j < len) {
        sv[i] = (double)ld_stream(val + j);
        sk[i] = ld_stream(crd2 + j);
        const int w = base >> 5;
        const uint32_t e = (uint32_t)lds_s32(w_ends + w * 4);
        if ((e >> x) & 1u) {
          int32_t f = f0 + lds_s32(w_rank + w * 4) + __popc(e & ((1u << x) - 1u));
          if (odd_fibers) f = fiber_of_end(j);
          sj[i] = __ldg(a.crd1 + f);
        }
      }
    }
  };
  auto store = [&](int half) {
#pragma unroll
    for (int i = 0; i < kPer; ++i) sts_entry(ring + (half * 32 + g + i * G) * 16, Entry16{sv[i], sk[i], sj[i]});
  };

  // ---- walk
  double tac[CPL];
  T q[kPF][CPL][1], prow[CPL][1];                // prow: the P row of the open slice
#pragma unroll
  for (int t = 0; t < CPL; ++t) tac[t] = 0.0;
  gather(pcol, ldp_bytes, __ldg(a.crd0 + s), prow);
  load(0);
  store(0);
  load(32);
  __syncwarp(mask);
#pragma unroll
  for (int u = 0; u < kPF; ++u) {
    int32_t ck, cj;
    lds_coords(ring + u * 16, ck, cj);
    gather(qcol, ldq_bytes, ck, q[u]);
  }
  int half = 0;
  bool last_ends = false;
  for (int32_t base = 0; base < len; base += 32, half ^= 1) {
    __syncwarp(mask);                            // every lane is done reading the half that is refilled next
    store(half ^ 1);
    __syncwarp(mask);
    load(base + 64);
    const int n = len - base < 32 ? len - base : 32;
    const uint32_t ends = (uint32_t)lds_s32(w_ends + (base >> 5) * 4), slices = (uint32_t)lds_s32(w_slices + (base >> 5) * 4);
    last_ends = (ends >> (n - 1)) & 1u;
#pragma unroll 1
    for (int e0 = 0; e0 < n; e0 += kPF) {
      const uint32_t ew = ends >> e0, sw = slices >> e0;
      const uint32_t at0 = ring + (half * 32 + e0) * 16, at1 = ring + ((half * 32 + e0 + kPF) & 63) * 16;
      if (n == 32 && (sw & ((1u << kPF) - 1u)) == 0) {       // the common case: no slice ends among these entries
        const uint32_t mine = CPL > 1 || ok[0] ? ew : 0u;
#pragma unroll
        for (int u = 0; u < kPF; ++u) {
          const Entry16 en = lds_entry(at0 + u * 16);
          double *const dst = a.acc + (int64_t)en.b * a.ldacc + col[0];
#pragma unroll
          for (int t = 0; t < CPL; ++t) {
            tac[t] = fma(en.v, (double)q[u][t][0], tac[t]);
            add_if(CPL == 1 || ok[t] ? mine & (1u << u) : 0u, t == 0 ? dst : dst + (col[t] - col[0]), tac[t], (double)prow[t][0]);
          }
          int32_t ck, cj;
          lds_coords(at1 + u * 16, ck, cj);
          gather(qcol, ldq_bytes, ck, q[u]);
        }
      } else {
#pragma unroll
        for (int u = 0; u < kPF; ++u) {
          if (e0 + u < n) {
            const double v = lds_f64(at0 + u * 16);
#pragma unroll
            for (int t = 0; t < CPL; ++t) tac[t] = fma(v, (double)q[u][t][0], tac[t]);
            if ((ew >> u) & 1u) {
              double *const dst = a.acc + (int64_t)lds_s32(at0 + u * 16 + 12) * a.ldacc;
#pragma unroll
              for (int t = 0; t < CPL; ++t) {
                if (ok[t]) atomicAdd(dst + col[t], tac[t] * (double)prow[t][0]);
                tac[t] = 0.0;
              }
              if (((sw >> u) & 1u) && next_slice(base + e0 + u)) gather(pcol, ldp_bytes, __ldg(a.crd0 + s), prow);
            }
            int32_t ck, cj;
            lds_coords(at1 + u * 16, ck, cj);
            gather(qcol, ldq_bytes, ck, q[u]);
          }
        }
      }
    }
  }
  if (!last_ends) {                              // a fiber that goes on in the next tile: its entries count by distributivity
    double *const dst = a.acc + (int64_t)__ldg(a.crd1 + f1) * a.ldacc;
#pragma unroll
    for (int t = 0; t < CPL; ++t)
      if (ok[t]) atomicAdd(dst + col[t], tac[t] * (double)prow[t][0]);
  }
}

// Six tiles per resident worker, or as many as the longest tiles make: how many adds a tile's fibers make, and into how popular
// rows, differs. One / two / three / four / six tiles: 3 M entries, R = 25, fp32 214 / 176 / 170 / 183 / 164 us; 7 M, R = 50 - / 613 /
// 591 / 575 / 561; 20 M, R = 32, fp64 four 805, six 787.
static int32_t level1_tile(int64_t N) {
  int64_t t = ceil_div(N, (int64_t)kSmCount * 4 * (kBlockThreads / 32) * 6);
  if (const char *e = getenv("COMET_TILE_ITEMS")) {
    const int v = atoi(e);
    if (v >= 8 && v <= (1 << 20)) t = v;
  }
  if (t < 32) t = 32;
  if (t > kLevel1Cap) t = kLevel1Cap;
  return (int32_t)align_up(t, 32);
}

size_t mttkrp_level1_bytes(int64_t N) {
  return 2 * align_up((size_t)(ceil_div(N > 0 ? N : 1, (int64_t)level1_tile(N)) + 1) * sizeof(int32_t), 256);
}

template <class T, int G, int CPL>
static void launch_level1(const Level1Args &a, cudaStream_t stream) {
  constexpr int WORKERS = kBlockThreads / G;
  mttkrp_level1_kernel<T, G, CPL><<<(unsigned)ceil_div(a.num_tiles, WORKERS), kBlockThreads, WORKERS * kLevel1WorkerBytes, stream>>>(a);
}

template <class T>
static comet_status_t level1_typed(Context *ctx, const Level1Args &base, int64_t R, cudaStream_t stream) {
  for (int64_t done = 0; done < R; done += 64) {
    Level1Args a = base;
    a.P = static_cast<const T *>(base.P) + done;
    a.Q = static_cast<const T *>(base.Q) + done;
    a.acc = base.acc + done;
    a.R = (int32_t)(R - done < 64 ? R - done : 64);
    if (a.R <= 16) launch_level1<T, 16, 1>(a, stream);
    else if (a.R <= 32) launch_level1<T, 32, 1>(a, stream);
    else launch_level1<T, 32, 2>(a, stream);
    COMET_LAUNCH_CHECK(ctx);
  }
  return COMET_OK;
}

comet_status_t mttkrp_level1(Context *ctx, int dtype, const int32_t *pos1, const int32_t *crd0, const int32_t *crd1,
                             const int32_t *pos2, const int32_t *crd2, const void *val, int64_t S, int64_t F, int64_t N,
                             const void *P, int64_t ldp, const void *Q, int64_t ldq, int64_t R, double *acc, int64_t ldacc,
                             char *part, cudaStream_t stream) {
  Level1Args a{};
  a.pos1 = pos1; a.crd0 = crd0; a.crd1 = crd1; a.seg_end2 = pos2 + 1; a.crd2 = crd2; a.val = val;
  a.S = S; a.F = F; a.N = N; a.P = P; a.ldp = ldp; a.Q = Q; a.ldq = ldq; a.acc = acc;
  a.ldacc = ldacc;
  a.tile = level1_tile(N);
  a.num_tiles = ceil_div(N, (int64_t)a.tile);
  int32_t *pf = (int32_t *)part, *ps = (int32_t *)(part + mttkrp_level1_bytes(N) / 2);
  level1_starts_kernel<<<(unsigned)ceil_div(a.num_tiles + 1, kBlockThreads), kBlockThreads, 0, stream>>>(a.seg_end2, pos1, S, F, N, a.tile,
                                                                                                        a.num_tiles, pf, ps);
  COMET_LAUNCH_CHECK(ctx);
  a.part_fiber = pf;
  a.part_slice = ps;
  return dtype == COMET_F32 ? level1_typed<float>(ctx, a, R, stream) : level1_typed<double>(ctx, a, R, stream);
}

}  // namespace comet

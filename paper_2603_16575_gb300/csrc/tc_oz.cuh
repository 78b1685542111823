// FP64 contraction on the tcgen05 tensor cores (sm_103a) by exact integer slices.
//
//   D[m][n] = sum_seg coef_seg sum_k A_seg[m][k] B_seg[n][k]      A, B, D in FP64
//
// FP64 runs at 2 FMAs a clock and SM on this part, BF16 tensor products at 4096: a
// product of integers cut small enough for the tensor core to sum them exactly gives an
// FP64 result from BF16 products (the splitting of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59 (2012) 95; integer form: Ootomo, Ozaki and Yokota, 2024).
//
//  * Within a chunk of CHUNK = 256 consecutive k, row m of A is
//      A[m][k] = 2^(e_m - 7) sum_{s=1..8} a_s 2^(-8 (s-1)),  a_s integer, |a_s| <= 128,
//    e_m the smallest exponent with max_k |A[m][k]| < 2^e_m (oz_split.cuh): 63 fractional
//    bits, ten more than the mantissa, so a value keeps its full mantissa down to 2^-10 of
//    the row's largest in the chunk and an absolute 2^(e_m - 64) below that.
//  * The mixed form takes five slices (39 bits, 15 products) or four (31 bits, 10 products).
//  * A product a_s b_t of level l = s + t is at most 2^14, a chunk sum of one slice pair at
//    most 2^22, and a sum of up to four pairs (levels 2-5) stays an exact FP32 integer
//    whatever the accumulator's rounding; levels 6-9 have 5 to 8 pairs, whose sums pass 2^24
//    only if every digit is extreme, and are 2^-32 and less of the result's scale then.
//    Levels above 9 (below 2^-64 of the chunk scale) are dropped: 36 products.
//  * The drain warps join the level sums of a chunk into one 64-bit integer (levels 2-7 by
//    shifts, 8 and 9 in full where it has room for them and rounded in otherwise), convert it once and add it to the FP64 sum of the element
//    with one FMA: K / 256 roundings per element where an FP64 dot product makes K.
//
// Bound: the multiplications (36 products: ~18k cycles an SM for 128 x 64 x 256) where K is a chunk or more, and
// the drain (FP64 and integer pipes; an FP64 operation holds the pipe of its sub-partition for 64 cycles a warp)
// below.  The eight 64-column level accumulators fill the 512 TMEM columns, so a tile is 64 columns wide (32 when
// it has no more); the drain of a chunk runs under the next chunk's MMAs: every level has its own full / empty
// barrier, so level l of the next chunk starts as soon as level l of this one has been read.
//
// Measured against the 64 x 64-tile FP64 CTA products (64 orbitals, 320 virtuals, 1200 aux): T_ii 8.5 ->
// 0.72 ms, projections 53.4 -> 3.0 ms, exchange blocks 16.9 -> 2.1 ms, S and F 2.9 -> 0.36 ms, digits
// included (one MMA a product: 0.80, 3.2, 2.6, 0.44); at 6 orbitals and 40 virtuals each is still faster or equal
// (T_ii 0.13 -> 0.05 ms), so there is no size rule.  The CUDA-core kernels remain for calls without room
// for the digits.
//
// Persistent CTAs (one per SM) over output tiles of 128 rows (TMEM lanes) x up to 64 columns:
//   warp 0     TMA producer: the slices of a 32-wide k-block, one box an operand, per stage (64-byte
//              swizzle, K-major), two stages of 96 KB
//   warp 1     TMEM allocation and the single MMA-issuing thread
//   warps 2-17 drain and epilogue: four warps per TMEM lane quarter, 16 columns each (the 64-bit
//              integers, the FP64 sums and the level being read of 32 columns do not fit the registers)
// Every mbarrier wait is bounded; a timeout sets ERR_TIMEOUT in *err, the roles leave their
// loops, the producer waits (bounded) for its copies in flight and the MMA thread for its
// last commit, and the CTA frees its tensor memory and returns without hanging.
#pragma once
#include <cuda.h>
#include <stdint.h>

#include <type_traits>

#include "oz_job.h"
#include "oz_split.cuh"
#include "tc_ptx.cuh"

namespace osv {
namespace oz {

constexpr int A_TILE = BM * BK * 2;          // 8 KB per A slice tile
constexpr int NDRAIN = 16;                   // drain warps
constexpr int DCOL = 16;                     // columns read at a time; four warps share a TMEM lane quarter
constexpr int NTHREADS = 64 + 32 * NDRAIN;
constexpr int KBC = CHUNK / BK;              // k-blocks of a full chunk
constexpr int TMEM_COLS = 512;
constexpr int ERR_TC_TIMEOUT = 16;           // same bit as ERR_TIMEOUT of the library

// Tensor maps of the two operands (k, row, slice): boxes of 32 k, every slice, and [0] half of or [1] all of a
// tile's rows.  One box takes an operand's part of a k-block: a TMA load costs ~95 cycles besides bytes / 80, so
// boxes of one slice and 64 or 32 rows (2 and 4 KB) fed the SM 17 to 29 bytes a cycle, these feed it 70 and more.
struct OzMaps {
  CUtensorMap a[2], b[2];
};

template <int NS>
struct Cfg {
  static constexpr int BN = tile_cols(NS);
  static constexpr int STAGE = NS * (A_TILE + BN * BK * 2);
  static constexpr int NSTAGE = NS == 8 ? 2 : 3;
  static constexpr int SMEM = NSTAGE * STAGE + 1024;   // + slack for 1024-byte alignment
  static constexpr int UNIT = 14 + 8 * (NS < 6 ? NS - 1 : 5);   // the joined integer is in units of 2^(e_m + e_n - UNIT)
};

// acc + coef * v * 2^x for the sum x of two chunk exponents less the integer's unit; out of the
// normal range: zero rows (EX_ZERO) add 0, non-finite rows (EX_NAN) give NaN, the rest in two factors.
__device__ __forceinline__ double pow2(int x) { return __longlong_as_double((long long)(x + 1023) << 52); }
__device__ __forceinline__ double oz_fma(long long v, int x, double coef, double acc) {
  if (x >= -1022 && x <= 1023) return fma((double)v, coef * pow2(x), acc);
  if (x >= EX_NAN / 2) return __longlong_as_double(0x7FF8000000000000ll);
  if (x < -2040 || x > 2040) return x < 0 ? acc : acc + (double)v * __longlong_as_double(0x7FF0000000000000ll);
  return fma(coef, (double)v * pow2(x / 2) * pow2(x - x / 2), acc);
}

// Columns of a tile's level accumulators, and rows of its B slices in shared memory: those of the widest, or half.
template <int NS>
__device__ __forceinline__ int width(const Job& jb) {
  return jb.n_valid <= tile_cols(NS) / 2 ? tile_cols(NS) / 2 : tile_cols(NS);
}
// Rows of its A slices in shared memory: with half of BM the MMAs read the next slice as the rows past the end.
__device__ __forceinline__ int height(const Job& jb) { return jb.m_valid <= BM / 2 ? BM / 2 : BM; }

// The products of one 16-wide k step (ks).  Slice sa of A times the slices 0 .. NS - 1 - sa of B adds to the levels
// sa .. NS - 1; those slices of B follow one another in shared memory as the levels do in TMEM, so one MMA takes as
// many of them as N = 256 holds: 12 MMAs for the 36 products of NS = 8, and A is read once for each.  (One MMA a
// product, N = 64, spent its time on the reads of A: 90 cycles for 32 of multiplication.)  free(l): level l of the
// last chunk has been read; done: barriers of the levels, committed as they become complete, or NULL.
template <int NS, int W, int H, class Free>
__device__ __forceinline__ bool issue(uint64_t da, uint64_t db, uint32_t dcol, int ks, bool zero, const Free& free,
                                      uint64_t* done) {
  constexpr int P = 256 / W;                                       // slices of B an MMA takes
  constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BM >> 4) << 24);
#pragma unroll
  for (int sa = 0; sa < NS; sa++) {
#pragma unroll
    for (int j = 0; j < NS - sa; j += P) {
      const int c = NS - sa - j < P ? NS - sa - j : P;
      if (sa == 0 && zero)
        for (int l = j; l < j + c; l++)
          if (!free(l)) return false;
      tc::mma_f16(dcol + (uint32_t)((sa + j) * W), da + (uint64_t)((sa * H * BK * 2 + 32 * ks) >> 4),
                  db + (uint64_t)((j * W * BK * 2 + 32 * ks) >> 4), idesc | ((uint32_t)(c * W >> 3) << 17),
                  sa == 0 && zero ? 0u : 1u);
    }
    if (done) tc::commit(done + sa);
  }
  return true;
}

// (ah, al) += (vh, vl) 2^x in FP32 pairs, the error terms gathered in al.
__device__ __forceinline__ void pair_add(float vh, float vl, int x, float& ah, float& al) {
  if (x < -120) return;                                            // zero rows, and terms below 2^-98
  float sc = __int_as_float((min(x, 127) + 127) << 23), t;
  if (x >= EX_NAN / 2) sc = __int_as_float(0x7FC00000);
  tc::two_sum(ah, vh * sc, ah, t);
  al += fmaf(vl, sc, t);
}

// Epi: epi(job, row, col0, acc) stores columns col0 .. col0 + 15 of the tile's row (row < m_valid); or, when
// Epi::kWarp, epi.warp(job, row, col0, acc) called by every lane of a drain warp, tiles without rows or columns
// for it included; or, when Epi::kDigits, epi.digits(job, row, col0, F) with F = round(value 2^(T - e)),
// T = epi.T, e = epi.exponent(job): a tile of one chunk comes there by an integer shift, never as an FP64 number;
// or, when Epi::kPair (NS <= 5), epi.pairs(job, row, col0, ah, al) with the sum as unnormalised FP32 pairs (the
// segments' coef is 1): the mixed form's products.  The FP64 drain takes three operations of an FP64 pipe that
// issues one warp in 64 cycles per element and chunk, more than the 15 products of a chunk; pairs take none.
// Epi::kLong: exponents are the epilogue's (one for each operand matrix), all segments add up in tensor memory (K up to
// ~1000: exact but for roundings at 2^-24 of a level in the later ones) and are read once, as pairs in units of the
// first level: epi.tile(job, epi.scale(job), row, col0, vh, vl) for the rows and columns of the tile.
template <int NS, class Epi>
__global__ void __launch_bounds__(NTHREADS, 1)
    k_oz(const __grid_constant__ OzMaps tm, const int* __restrict__ exA,
         const int* __restrict__ exB, const Job* __restrict__ jobs, int n_jobs, const Seg* __restrict__ segs,
         const int* __restrict__ skip, int* err, Epi epi) {
  using C = Cfg<NS>;
  constexpr int NST = C::NSTAGE, BN = C::BN;
  extern __shared__ uint8_t dsm[];
  __shared__ __align__(8) uint64_t bar_full[NST], bar_empty[NST], bar_accf[NS], bar_acce[NS];
  __shared__ uint32_t s_tmem;
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dsm) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = tc::su32(sm);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::su32(&s_tmem)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; s++) {
      tc::mbar_init(&bar_full[s], 1);
      tc::mbar_init(&bar_empty[s], 1);
    }
    for (int l = 0; l < NS; l++) {
      tc::mbar_init(&bar_accf[l], 1);
      tc::mbar_init(&bar_acce[l], NDRAIN);
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
    for (int u = 0; u < 2; u++) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm.a[u])) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm.b[u])) : "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = s_tmem;
  bool ok = true;
  // The CTA takes tiles blockIdx.x, + gridDim.x, ...; g counts its k-blocks and ch its
  // chunks, so all barrier phases carry over from tile to tile.  Every role walks the same
  // (tile, segment, chunk, k-block) sequence.
  if (warp == 0) {
    if (lane == 0) {                                             // ---- TMA producer
      long long g = 0;
      for (int tile = blockIdx.x; ok && tile < n_jobs; tile += gridDim.x) {
        const Job jb = jobs[tile];
        if (jb.skip >= 0 && skip[jb.skip]) continue;
        const int h = height(jb), w = width<NS>(jb);
        const uint32_t bytes = NS * (h + w) * BK * 2;
        const CUtensorMap *ma = &tm.a[h == BM], *mb = &tm.b[w == BN];
        for (int q = 0; ok && q < jb.nseg; q++) {
          const Seg sg = segs[jb.seg0 + q];
          const int nkb = (sg.K + BK - 1) / BK, ra = sg.a.row + jb.m0, rb = sg.b.row + jb.n0;
          for (int c = 0; c < nkb; c++, g++) {
            const int s = (int)(g % NST);
            if (g >= NST) ok = tc::mbar_wait(tc::su32(&bar_empty[s]), (uint32_t)(((g / NST) - 1) & 1));
            if (!ok) break;
            const uint32_t fb = tc::su32(&bar_full[s]);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(bytes) : "memory");
            const uint32_t st = sbase + s * C::STAGE;
            tc::tma_load_3d(st, ma, fb, c * BK, ra, 0);
            tc::tma_load_3d(st + NS * A_TILE, mb, fb, c * BK, rb, 0);
          }
        }
      }
      if (!ok) {
        // leaving early: let the copies already issued land first (bounded waits); only the
        // last armed k-block of each stage can be outstanding
        for (long long gg = g - 1; gg >= 0 && gg >= g - NST; gg--)
          tc::mbar_wait(tc::su32(&bar_full[gg % NST]), (uint32_t)((gg / NST) & 1));
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {                                             // ---- MMA issuer
      long long g = 0, ch = 0;
      bool was_wide = true;
      for (int tile = blockIdx.x; ok && tile < n_jobs; tile += gridDim.x) {
        const Job jb = jobs[tile];
        if (jb.skip >= 0 && skip[jb.skip]) continue;
        const bool wide = width<NS>(jb) == BN, tall = height(jb) == BM;
        for (int q = 0; ok && q < jb.nseg; q++) {
          const int K = segs[jb.seg0 + q].K, nkb = (K + BK - 1) / BK;
          for (int c = 0; c < nkb; c++, g++) {
            const int s = (int)(g % NST);
            bool first = (c % KBC) == 0, last = (c % KBC) == KBC - 1 || c == nkb - 1;
            if constexpr (Epi::kLong) {
              first = q == 0 && c == 0;
              last = q == jb.nseg - 1 && c == nkb - 1;
            }
            const int nks = K - c * BK > 16 ? 2 : 1;             // 16-wide steps that hold elements
            ok = tc::mbar_wait(tc::su32(&bar_full[s]), (uint32_t)((g / NST) & 1));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t st = sbase + s * C::STAGE;
            const uint64_t da = tc::desc_sw64(st), db = tc::desc_sw64(st + NS * A_TILE);
            auto level_free = [&](int l) {
              if (ch < 1) return true;
              const bool f = tc::mbar_wait(tc::su32(&bar_acce[l]), (uint32_t)((ch - 1) & 1));
              asm volatile("tcgen05.fence::after_thread_sync;");
              return f;
            };
            if (first && wide != was_wide) {                     // the levels lie elsewhere: all of the last chunk first
              for (int l = 0; ok && l < NS; l++) ok = level_free(l);
              if (!ok) break;
              was_wide = wide;
            }
            for (int ks = 0; ks < nks; ks++) {
              const bool fin = last && ks == nks - 1;
              auto go = [&](auto W, auto H) {
                return issue<NS, W, H>(da, db, tmem, ks, first && ks == 0, level_free, fin ? bar_accf : nullptr);
              };
              if (wide)
                ok = tall ? go(std::integral_constant<int, BN>{}, std::integral_constant<int, BM>{})
                          : go(std::integral_constant<int, BN>{}, std::integral_constant<int, BM / 2>{});
              else
                ok = tall ? go(std::integral_constant<int, BN / 2>{}, std::integral_constant<int, BM>{})
                          : go(std::integral_constant<int, BN / 2>{}, std::integral_constant<int, BM / 2>{});
              if (!ok) break;
            }
            if (!ok) break;
            tc::commit(&bar_empty[s]);
            if (last) ch++;
          }
        }
      }
      // wait (bounded) for the last commit of each stage: every MMA issued has then completed
      // and no arrival is in flight when the CTA exits
      if (!ok) {
        tc::commit(&bar_empty[g % NST]);
        g++;
      }
      for (long long gg = g - 1; gg >= 0 && gg >= g - NST; gg--)
        tc::mbar_wait(tc::su32(&bar_empty[gg % NST]), (uint32_t)((gg / NST) & 1));
    }
  } else {                                                       // ---- drain + epilogue
    const int quad = warp & 3;                                   // TMEM lane quarter of this warp
    const int col0 = ((warp - 2) >> 2) * (BN / 4);               // and its columns
    const uint32_t lcol = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)col0;
    const int row = 32 * quad + lane;
    long long ch = 0;
    for (int tile = blockIdx.x; ok && tile < n_jobs; tile += gridDim.x) {
      const Job jb = jobs[tile];
      if (jb.skip >= 0 && skip[jb.skip]) continue;
      const bool live = col0 < jb.n_valid && 32 * quad < jb.m_valid;   // warp-uniform
      const int w = width<NS>(jb);
      if constexpr (Epi::kLong) {
        // one sum over all segments, read DCOL columns at a time
        typename Epi::Scale sc = epi.scale(jb);
#pragma unroll
        for (int g = 0; g < BN / 4; g += DCOL) {
          const bool here = col0 + g < jb.n_valid && 32 * quad < jb.m_valid;   // warp-uniform
          float vh[DCOL], vl[DCOL];
#pragma unroll
          for (int l = 0; l < NS; l++) {
            if (g == 0) {
              ok = __all_sync(0xffffffffu, tc::mbar_wait(tc::su32(&bar_accf[l]), (uint32_t)(ch & 1)));
              if (!ok) break;
              asm volatile("tcgen05.fence::after_thread_sync;");
            }
            uint32_t x[DCOL];
            if (here) {
              OSV_TMEM_LD16(lcol + l * w + g, x);
              asm volatile("tcgen05.wait::ld.sync.aligned;");
            }
            if (g == BN / 4 - DCOL) {
              asm volatile("tcgen05.fence::before_thread_sync;");
              __syncwarp();
              if (lane == 0) tc::mbar_arrive(&bar_acce[l]);
            }
            if (!here) continue;
#pragma unroll
            for (int u = 0; u < DCOL; u++) {
              const float y = __uint_as_float(x[u]) * __int_as_float((127 - 8 * l) << 23);
              if (l == 0) { vh[u] = y; vl[u] = 0.f; }
              else if (l == 1) tc::two_sum(vh[u], y, vh[u], vl[u]);
              else vl[u] += y;
            }
          }
          if (!ok) break;
          if (here && row < jb.m_valid) epi.tile(jb, sc, row, col0 + g, vh, vl);
        }
        if (!ok) break;
        ch++;
        continue;
      }
      double acc[Epi::kDigits || Epi::kPair ? 1 : DCOL];
      float ah[Epi::kPair ? DCOL : 1], al[Epi::kPair ? DCOL : 1];
      long long f[Epi::kDigits ? DCOL : 1];
      int eout = 0;
      if constexpr (Epi::kDigits) {
        eout = epi.exponent(jb);
#pragma unroll
        for (int u = 0; u < DCOL; u++) f[u] = 0;
      } else if constexpr (Epi::kPair) {
#pragma unroll
        for (int u = 0; u < DCOL; u++) ah[u] = al[u] = 0.f;
      } else {
#pragma unroll
        for (int u = 0; u < DCOL; u++) acc[u] = 0.0;
      }
      for (int q = 0; ok && q < jb.nseg; q++) {
        const Seg* sg = segs + jb.seg0 + q;
        const int nch = (sg->K + CHUNK - 1) / CHUNK;
        const int* ea_p = exA + sg->a.eb + (long long)(jb.m0 + min(row, jb.m_valid - 1)) * sg->a.es;
        const int* eb_p = exB + sg->b.eb + (long long)(jb.n0 + min(col0 + (lane & (DCOL - 1)), jb.n_valid - 1)) * sg->b.es;
        const double coef = sg->coef;
        for (int c = 0; ok && c < nch; c++, ch++) {
          const uint32_t ph = (uint32_t)(ch & 1);
          const int ea = ea_p[c] - C::UNIT, eb = eb_p[c];
          long long v[Epi::kPair ? 1 : DCOL];
          float vh[Epi::kPair ? DCOL : 1], vl[Epi::kPair ? DCOL : 1];
          int lo[NS > 6 ? DCOL : 1];
          if constexpr (!Epi::kPair) {
#pragma unroll
            for (int u = 0; u < DCOL; u++) v[u] = 0;
          }
#pragma unroll
          for (int l = 0; l < NS; l++) {
            ok = __all_sync(0xffffffffu, tc::mbar_wait(tc::su32(&bar_accf[l]), ph));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            uint32_t x[DCOL];
            if (live) {
              OSV_TMEM_LD16(lcol + l * w, x);
              asm volatile("tcgen05.wait::ld.sync.aligned;");
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&bar_acce[l]);
            if (!live) continue;
#pragma unroll
            for (int u = 0; u < DCOL; u++) {
              if constexpr (Epi::kPair) {                            // levels as an FP32 pair in units of the first
                const float y = __uint_as_float(x[u]) * __int_as_float((127 - 8 * l) << 23);
                if (l == 0) { vh[u] = y; vl[u] = 0.f; }
                else if (l == 1) tc::two_sum(vh[u], y, vh[u], vl[u]);
                else vl[u] += y;
                if (l == NS - 1) pair_add(vh[u], vl[u], ea + __shfl_sync(0xffffffffu, eb, u) + C::UNIT - 14, ah[u], al[u]);
                continue;
              }
              const int d = __float2int_rn(__uint_as_float(x[u]));
              if (l < 6) v[u] = (v[u] << 8) + d;                   // levels 2 .. 7
              if constexpr (NS > 6) {
                if (l == 6) lo[u] = d;                             // level 8, unit 2^-8
              }
              if (l == NS - 1) {                                   // the chunk is complete
                int e = ea + __shfl_sync(0xffffffffu, eb, u);
                long long t = v[u];
                if constexpr (NS > 6) {                            // level 9, unit 2^-16
                  const long long w = ((long long)lo[u] << 8) + d;
                  if ((unsigned long long)(t + (1ll << 45)) >> 46) t += (w + 32768) >> 16;
                  else {                                           // room below: levels 8 and 9 in full
                    t = (t << 16) + w;
                    e -= 16;
                  }
                }
                if constexpr (Epi::kDigits) {
                  // F = t 2^(e + T - eout), rounded; |F| < 2^T since eout is a bound of the value
                  const int sh = eout - Epi::T - e;
                  f[u] += sh <= 0 ? (sh > -63 ? t << -sh : 0) : (sh < 63 ? (t + (1ll << (sh - 1))) >> sh : 0);
                } else {
                  acc[u] = oz_fma(t, e, coef, acc[u]);
                }
              }
            }
          }
        }
      }
      if (!ok) break;
      if constexpr (Epi::kDigits) {
        if (row < jb.m_valid && live) epi.digits(jb, row, col0, f);
      } else if constexpr (Epi::kLong) {                            // (stored above)
      } else if constexpr (Epi::kPair) {
        if (row < jb.m_valid && live) epi.pairs(jb, row, col0, ah, al);
      } else if constexpr (Epi::kWarp) {
        epi.warp(jb, row, col0, acc);
      } else {
        if (row < jb.m_valid && live) epi(jb, row, col0, acc);
      }
    }
  }
  if (!ok) atomicOr(err, ERR_TC_TIMEOUT);
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
}

}  // namespace oz
}  // namespace osv

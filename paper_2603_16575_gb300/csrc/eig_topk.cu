// Householder tridiagonalisation on a thread-block cluster per matrix, and the eigenpairs
// above a threshold from it (Eq. osv_gen), for matrices of order > EIG_FULL_MAX.
//
// Bound: FP64 arithmetic of the sweep (four FMAs per element of the trailing lower
// triangle and step, 2 FMAs a clock and SM) at a few hundred rows and more, the latency of
// a step (three CTA-wide scalar reductions and one exchange of vectors) below.  One CTA
// per matrix leaves SMs idle when there are fewer matrices than SMs and pays the L2 round
// trip of the matrix on every step, so a cluster of up to eight CTAs shares a matrix:
//  * the lower triangle is cut into 32 x 32 tiles counted from the END of the matrix, so that
//    the tiles still alive after step k are the first ones; tile t belongs to CTA t mod C
//    for the whole reduction and stays in its shared memory as far as that reaches (the
//    first tiles, which live longest); the others stay in global memory (L2);
//  * a step applies the previous rank-2 update and forms the tile's part of A v in one pass;
//    the parts and the next column go to a global buffer (two, alternating), one cluster
//    barrier follows, and every CTA forms the vectors of the step from the buffer
//    in the same fixed order, so the result does not depend on timing.
// Few alive tiles are cut into two or four parts, a warp each.
//
// An FP64 operation of a warp holds its sub-partition's pipe for 64 cycles whatever else is in flight, so on
// the critical path their number counts: the scalars of a reflector are formed by one lane with a dozen
// operations (reflector), and nothing is computed redundantly by every warp.
//
// Measured against one CTA per matrix for the whole of it (reduction, eigenvalues by Sturm counts with a
// division a row, a warp's Gram-Schmidt per cluster): 24 matrices of order 760 470 -> 43 ms (the reduction 89 -> 26, at
// 5 CTAs), 48 of 243 12.5 -> 5.2 (5.9 -> 3.5, 2 CTAs), 64 of 320 19.9 -> 8.3 (2 CTAs), 32 of 160 7.0 -> 2.2
// (4 CTAs), 6 of 40 1.2 -> 0.5 (6 CTAs); double-float, 64 of 320 9.6 -> 6.9 (2 CTAs), 128 of 640 39 -> 40 (1 CTA).
#include <algorithm>
#include <cmath>

#include "eig.cuh"
#include "eig_topk.h"
#include "internal.h"

namespace osv {
namespace {

constexpr int TD_TILE = 32 * 33;           // elements of a resident tile (padded rows)
constexpr int TD_STAGE = 8 * 33;           // elements of a warp's staging rows (tiles in global memory)
constexpr size_t TD_SMEM = 227 * 1024 - 1024;   // dynamic shared memory; the rest is static
constexpr double OR_TOL = 1e-6;            // gap (of ||T||) below which vectors are orthogonalised by Gram-Schmidt

// The arithmetic of the reduction: FP64, or double-float pairs (same size) for the mixed form.
struct ArD {
  using E = double;
  static constexpr int NTH = 512;          // threads of a CTA
  static constexpr int NWS = 16;           // sweeping warps at most
  static constexpr bool DF = false;
  static constexpr int SPREAD = 32;        // alive tiles per CTA below which they are cut into parts
  struct Acc {
    double s = 0.0;
    __device__ __forceinline__ void fma(E a, E b) { s = ::fma(a, b, s); }
    __device__ __forceinline__ E get() const { return s; }
  };
  static __device__ __forceinline__ E zero() { return 0.0; }
  static __device__ __forceinline__ E one() { return 1.0; }
  static __device__ __forceinline__ E from(double x) { return x; }
  static __device__ __forceinline__ double to(E x) { return x; }
  static __device__ __forceinline__ E neg(E x) { return -x; }
  static __device__ __forceinline__ E add(E a, E b) { return a + b; }
  static __device__ __forceinline__ E mul(E a, E b) { return a * b; }
  static __device__ __forceinline__ E fma1(E x, E y, E a) { return ::fma(x, y, a); }
  static __device__ __forceinline__ E fma2(E x1, E y1, E x2, E y2, E a) { return ::fma(x1, y1, ::fma(x2, y2, a)); }
  static __device__ __forceinline__ E sx(E a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
  static __device__ __forceinline__ E ld(const E* p) { return __ldcg(p); }
  static __device__ __forceinline__ void st(E* p, E v) { __stcg(p, v); }
  static __device__ __forceinline__ void factor(const E* d, const E* e, int n, double lam, double small, E* ui, E* u1,
                                                E* u2, E* mul, int* piv) {
    tri_factor_lanes(d, e, n, lam, small, ui, u1, u2, mul, piv);
  }
  // the scale of the next read, from this solve
  static __device__ __forceinline__ double solve(int n, double sc, const E* ui, const E* u1, const E* u2, const E* mul,
                                                 const int* piv, E* y) {
    const double nn = tri_solve_lanes(n, sc, ui, u1, u2, mul, piv, y);
    return nn > 0.0 ? 1.0 / sqrt(nn) : 0.0;
  }
};
struct ArF {
  using E = dfl;
  static constexpr int NTH = 1024;
  static constexpr int NWS = 32;
  static constexpr bool DF = true;
  static constexpr int SPREAD = 48;
  struct Acc {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void fma(E a, E b) { df_acc(h, l, a, b); }
    __device__ __forceinline__ E get() const { return df_norm(h, l); }
  };
  static __device__ __forceinline__ E zero() { return dfl{0.f, 0.f}; }
  static __device__ __forceinline__ E one() { return dfl{1.f, 0.f}; }
  static __device__ __forceinline__ E from(double x) { return df_from(x); }
  static __device__ __forceinline__ double to(E x) { return df_to(x); }
  static __device__ __forceinline__ E neg(E x) { return df_neg(x); }
  static __device__ __forceinline__ E add(E a, E b) { return df_add(a, b); }
  static __device__ __forceinline__ E mul(E a, E b) { return df_mul(a, b); }
  static __device__ __forceinline__ E fma1(E x, E y, E a) { return df_fma1(x, y, a); }
  static __device__ __forceinline__ E fma2(E x1, E y1, E x2, E y2, E a) { return df_fma2(x1, y1, x2, y2, a); }
  static __device__ __forceinline__ E sx(E a, int o) { return df_shfl_xor(a, o); }
  static __device__ __forceinline__ E ld(const E* p) {
    const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
    return dfl{v.x, v.y};
  }
  static __device__ __forceinline__ void st(E* p, E v) { __stcg(reinterpret_cast<float2*>(p), make_float2(v.h, v.l)); }
  static __device__ __forceinline__ void factor(const E* d, const E* e, int n, double lam, double small, E* ui, E* u1,
                                                E* u2, E* mul, int* piv) {
    tri_factor_lanes_df(d, e, n, df_from(lam), (float)small, ui, u1, u2, mul, piv);
  }
  static __device__ __forceinline__ double solve(int n, double sc, const E* ui, const E* u1, const E* u2, const E* mul,
                                                 const int* piv, E* y) {
    const float am = tri_solve_lanes_df(n, (float)sc, ui, u1, u2, mul, piv, y);
    return am > 0.f ? (double)(1.f / am) : 0.0;
  }
};

__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Scalars of the reflector of (alpha, x), sigma = |x|^2: beta = -+ sqrt(alpha^2 + sigma),
// tu = (beta - alpha) / beta, sc = 1 / (alpha - beta).  An FP64 operation holds the pipe for 64 cycles, a
// square root or division ten of them, on the critical path of every step: the FP32 reciprocal (root) of the
// mantissa refined by one step of third order (Halley; error ~2^-60 before rounding) takes six.
__device__ __forceinline__ void reflector(double alpha, double sigma, double& beta, double& tu, double& sc) {
  const double s = fma(alpha, alpha, sigma);
  const int hi = __double2hiint(s), lo = __double2loint(s), ex = (hi >> 20) & 2047;
  const bool neg = alpha <= 0.0;
  if (ex < 64 || ex > 1983) {   // zero, near the ends of the range, not finite
    const double mu = sqrt(s);
    beta = neg ? mu : -mu;
    tu = (beta - alpha) / beta;
    sc = 1.0 / (alpha - beta);
    return;
  }
  const int q = (ex - 1023) >> 1;                                  // s = m 4^q, m in [1, 4)
  const double m = __hiloint2double(hi - (q << 21), lo);
  const double r0 = widen(rsqrtf(mant_f(hi - (q << 21), lo)), 0);
  const double e = fma(-m * r0, r0, 1.0);
  const double r = fma(r0 * e, fma(e, 0.375, 0.5), r0);            // m^(-1/2)
  const double mr = m * r;
  const double mu = __hiloint2double(__double2hiint(mr) + (q << 20), __double2loint(mr));
  const double ri = __hiloint2double(__double2hiint(r) - (q << 20), __double2loint(r));
  beta = neg ? mu : -mu;
  tu = fma(fabs(alpha), ri, 1.0);
  const double x = fabs(alpha) + mu;                               // |alpha - beta|, in [mu, 2 mu]
  const int xh = __double2hiint(x), xl = __double2loint(x), xe = (xh >> 20) - 1023;
  const double xm = __hiloint2double(xh - (xe << 20), xl);
  const double y0 = widen(__frcp_rn(mant_f(xh - (xe << 20), xl)), 0);
  const double d = fma(-xm, y0, 1.0);
  const double y = fma(y0, fma(d, d, d), y0);
  const double ya = __hiloint2double(__double2hiint(y) - (xe << 20), __double2loint(y));
  sc = neg ? -ya : ya;
}

template <class R>
__device__ __forceinline__ typename R::E warp_add(typename R::E v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = R::add(v, R::sx(v, o));
  return v;
}

// sum_i x[i] y[i], i < m, by one warp (fixed order)
template <class R>
__device__ __forceinline__ typename R::E warp_dot(const typename R::E* x, const typename R::E* y, int m) {
  const int lane = threadIdx.x & 31;
  typename R::Acc a, b;
  int i = lane;
  for (; i + 32 < m; i += 64) {
    a.fma(x[i], y[i]);
    b.fma(x[i + 32], y[i + 32]);
  }
  if (i < m) a.fma(x[i], y[i]);
  return warp_add<R>(R::add(a.get(), b.get()));
}

// Room of one exchange buffer: column parts, row parts, next column.
__host__ __device__ inline size_t td_buf(int n) {
  const size_t nb = (n + 31) / 32;
  return 5 * nb * 32 * nb + 32 * nb;
}

// Eight rows of a tile (rows: their 33-padded place in shared memory, resident or staged; index of the first: ri)
// receive the previous update; col += their part of the column sums.  EDGE: the tile is on the diagonal or
// past the end in its columns, and elements outside become zero.
template <class R, bool EDGE>
__device__ __forceinline__ void sweep_rows(typename R::E* rows, typename R::E* g, int n, bool res, int ri, int ci, int L,
                                           typename R::E nvc, typename R::E nwc, const typename R::E* vp,
                                           const typename R::E* wp, const typename R::E* vk, typename R::Acc& col) {
  using E = typename R::E;
  const int lane = threadIdx.x & 31;
  E av[8];
  if (res) {
#pragma unroll
    for (int u = 0; u < 8; u++) av[u] = rows[u * 33 + lane];
  } else {
#pragma unroll
    for (int u = 0; u < 8; u++)
      av[u] = !EDGE || (ci < L && ri + u <= ci) ? R::ld(g - (ptrdiff_t)u * n) : R::zero();
  }
#pragma unroll
  for (int u = 0; u < 8; u++) {
    E a = R::fma2(vp[ri + u], nwc, wp[ri + u], nvc, av[u]);
    if (EDGE && !(ci < L && ri + u <= ci)) a = R::zero();
    else if (!res) R::st(g - (ptrdiff_t)u * n, a);
    col.fma(a, vk[ri + u]);
    rows[u * 33 + lane] = a;
  }
}

// Tridiagonalise A (n x n, row-major, lower triangle read) with the C CTAs of this cluster, rank
// `rank`: d[n], e[n-1], tau[n], reflector k in row k to the right of the diagonal
// (A[k][k+1+t] = v_t, v_0 = 1; pairs when refl_df).  Index i below is n - 1 - (row or column).
// vp, wp, vk: 32 ceil(n/32) elements of shared memory each; tiles: cap resident tiles;
// stage: nsw x TD_STAGE elements (unused when every tile is resident).  part: 2 td_buf(n) elements.
template <class R>
__device__ void tridiag_cluster(double* A, int n, double* d, double* e, double* tau, typename R::E* vp,
                                typename R::E* wp, typename R::E* vk, typename R::E* tiles, int cap,
                                typename R::E* stage, int nsw, typename R::E* part, bool refl_df, int rank, int C) {
  using E = typename R::E;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nb0 = (n + 31) >> 5, npad = 32 * nb0;
  E* Ad = reinterpret_cast<E*>(A);
  __shared__ E s_tk, s_hk, s_sc, s_pl, s_K, s_nwl;
  __shared__ bool s_nz;
  // column 0 before any element is converted
  for (int i = tid; i < npad; i += R::NTH) {
    vp[i] = R::zero();
    wp[i] = R::zero();
    const E a = i < n ? R::from(A[(size_t)(n - 1 - i) * n]) : R::zero();
    vk[i] = a;
    if (rank == 0 && i == n - 1) d[0] = R::to(a);
  }
  cluster_sync();
  const int nt0 = nb0 * (nb0 + 1) / 2;
  for (int t = rank + C * warp; t < nt0; t += C * (R::NTH / 32)) {
    int cb = 0;
    while ((cb + 1) * (cb + 2) / 2 <= t) cb++;
    const int rb = t - cb * (cb + 1) / 2, slot = t / C, ci = 32 * cb + lane;
    if (slot < cap) {
      E* tl = tiles + (size_t)slot * TD_TILE;
      for (int r = 0; r < 32; r++) {
        const int ri = 32 * rb + r;
        tl[r * 33 + lane] = (ri <= ci && ci < n) ? R::from(A[(size_t)(n - 1 - ri) * n + (n - 1 - ci)]) : R::zero();
      }
    } else if (R::DF) {
      for (int r = 0; r < 32; r++) {
        const int ri = 32 * rb + r;
        if (ri <= ci && ci < n) {
          const size_t at = (size_t)(n - 1 - ri) * n + (n - 1 - ci);
          R::st(Ad + at, R::from(A[at]));
        }
      }
    }
  }
  __syncthreads();
  for (int k = 0; k + 2 < n; k++) {
    const int L = n - 1 - k;   // trailing indices 0 .. L-1; vk holds column k
    // Householder reflector of column k (scalars in FP64)
    if (warp == 0) {
      const double sigma = R::to(warp_dot<R>(vk, vk, L - 1));
      if (lane == 0) {
        const double alpha = R::to(vk[L - 1]);
        const bool nz = sigma > 0.0;
        double tu = 0.0, beta = alpha, sc = 0.0;
        if (nz) reflector(alpha, sigma, beta, tu, sc);
        s_nz = nz;
        s_tk = R::from(tu);
        s_hk = R::from(-0.5 * tu);
        s_sc = R::from(sc);
        if (rank == 0) {
          e[k] = beta;
          tau[k] = tu;
        }
      }
    }
    __syncthreads();
    const bool nz = s_nz;
    const E sc = s_sc, tk = s_tk;
    const int nb = (L + 31) >> 5, ntile = nb * (nb + 1) / 2;
    for (int i = tid; i < 32 * nb; i += R::NTH) {
      const E v = i < L - 1 ? R::mul(vk[i], sc) : (i == L - 1 ? R::one() : R::zero());
      vk[i] = nz ? v : R::zero();
      if (rank == 0 && i < L) {
        const size_t at = (size_t)k * n + (n - 1 - i);
        if (refl_df) Ad[at] = v;
        else A[at] = R::to(v);
      }
    }
    __syncthreads();
    // previous update and parts of A v, tile by tile
    E* buf = part + (size_t)(k & 1) * td_buf(n);
    E* gcol = buf;
    E* grow = buf + (size_t)4 * nb0 * npad;
    E* gnext = grow + (size_t)nb0 * npad;
    const int np = ntile >= R::SPREAD * C ? 1 : (2 * ntile >= R::SPREAD * C ? 2 : 4);
    const int nloc = (ntile - rank + C - 1) / C, pr = 32 / np;   // parts of pr rows
    for (int it = warp; it < nloc * np && warp < nsw; it += nsw) {
      const int slot = it / np, pt = it % np, t = slot * C + rank;
      int cb = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
      while ((cb + 1) * (cb + 2) / 2 <= t) cb++;
      while (cb * (cb + 1) / 2 > t) cb--;
      const int rb = t - cb * (cb + 1) / 2, ci = 32 * cb + lane;
      const bool res = slot < cap, diag = rb == cb, edge = diag || 32 * cb + 32 > L;
      E* tl = res ? tiles + (size_t)slot * TD_TILE : stage + (size_t)warp * TD_STAGE;
      const E nvc = R::neg(vp[ci]), nwc = R::neg(wp[ci]);
      const int r8 = lane & 7, g8 = 8 * (lane >> 3);   // row sums: lane (g, r) sums a quarter of row r
      E vc[8];
#pragma unroll
      for (int j = 0; j < 8; j++) vc[j] = vk[32 * cb + g8 + j];
      typename R::Acc col;
      for (int q = pr * pt; q < pr * pt + pr; q += 8) {
        E* rows = res ? tl + q * 33 : tl;
        const int ri = 32 * rb + q;
        E* g = Ad + (ptrdiff_t)(n - 1 - ri) * n + (n - 1 - ci);   // not followed outside the matrix
        if (edge) sweep_rows<R, true>(rows, g, n, res, ri, ci, L, nvc, nwc, vp, wp, vk, col);
        else sweep_rows<R, false>(rows, g, n, res, ri, ci, L, nvc, nwc, vp, wp, vk, col);
        __syncwarp();
        if (cb == nb - 1 && lane < 8 && ri + lane < L) R::st(gnext + ri + lane, rows[lane * 33 + L - 1 - 32 * cb]);
        typename R::Acc row;
#pragma unroll
        for (int j = 0; j < 8; j++) {
          E x = rows[r8 * 33 + g8 + j];
          if (diag && q + r8 == g8 + j) x = R::zero();   // the strictly lower part
          row.fma(x, vc[j]);
        }
        E rs = row.get();
        rs = R::add(rs, R::sx(rs, 8));
        rs = R::add(rs, R::sx(rs, 16));
        if (lane < 8) R::st(grow + (size_t)cb * npad + ri + lane, rs);
        __syncwarp();
      }
      R::st(gcol + (size_t)(np * rb + pt) * npad + ci, col.get());
    }
    cluster_sync();
    const bool more = k + 3 < n;
    const E next = more && tid < L ? R::ld(gnext + tid) : R::zero();   // of the column below, under the sums
    // p = tau A v from the parts, then w = p - (tau / 2)(p . v) v; G lanes share the terms of an element
    const int G = L <= R::NTH / 4 ? 4 : (L <= R::NTH / 2 ? 2 : 1), W = 32 / G;
    for (int i0 = warp * W; i0 < L; i0 += (R::NTH / 32) * W) {
      const int i = i0 + lane % W, g = lane / W, b = i >> 5;
      E s = R::zero();
      if (i < L) {   // four loads (L2) in flight before their sums
        for (int j0 = g; j0 < np * (b + 1); j0 += 4 * G) {
          E x[4];
#pragma unroll
          for (int u = 0; u < 4; u++)
            x[u] = j0 + u * G < np * (b + 1) ? R::ld(gcol + (size_t)(j0 + u * G) * npad + i) : R::zero();
          s = R::add(s, R::add(R::add(x[0], x[1]), R::add(x[2], x[3])));
        }
        for (int j0 = b + g; j0 < nb; j0 += 4 * G) {
          E x[4];
#pragma unroll
          for (int u = 0; u < 4; u++)
            x[u] = j0 + u * G < nb ? R::ld(grow + (size_t)(j0 + u * G) * npad + i) : R::zero();
          s = R::add(s, R::add(R::add(x[0], x[1]), R::add(x[2], x[3])));
        }
      }
      for (int o = W; o < 32; o <<= 1) s = R::add(s, R::sx(s, o));
      if (i < L && g == 0) {
        s = R::mul(s, tk);
        wp[i] = s;
        if (i == L - 1) s_pl = s;
      }
    }
    __syncthreads();
    if (warp == 0) {
      const E pv = warp_dot<R>(wp, vk, L);
      if (lane == 0) {
        const E nK = R::mul(s_hk, pv);
        s_K = nK;
        s_nwl = R::neg(nz ? R::add(nK, s_pl) : s_pl);   // -w of the next column's row (v = 1 there)
      }
    }
    __syncthreads();
    // w, and column k + 1 with this step's update
    const E nK = s_K, nwl = s_nwl, nvl = nz ? R::neg(R::one()) : R::zero();
    for (int i = tid; i < L; i += R::NTH) {
      const E v = vk[i], w = R::fma1(nK, v, wp[i]);
      wp[i] = w;
      vp[i] = v;
      if (more) {
        const E a = R::fma2(v, nwl, w, nvl, i == tid ? next : R::ld(gnext + i));
        if (i < L - 1) vk[i] = a;
        else if (rank == 0) d[k + 1] = R::to(a);
      }
    }
    __syncthreads();
  }
  // the trailing 2 x 2 block (in tile 0) receives the last update
  if (rank == 0 && tid == 0) {
    auto at = [&](int ri, int ci) {
      return R::to(cap > 0 ? tiles[ri * 33 + ci] : Ad[(size_t)(n - 1 - ri) * n + (n - 1 - ci)]);
    };
    double x00 = at(1, 1), x10 = at(0, 1), x11 = at(0, 0);
    const double v0 = R::to(vp[1]), v1 = R::to(vp[0]), w0 = R::to(wp[1]), w1 = R::to(wp[0]);
    x00 -= 2.0 * v0 * w0;
    x10 -= v1 * w0 + w1 * v0;
    x11 -= 2.0 * v1 * w1;
    d[n - 2] = x00;
    e[n - 2] = x10;
    d[n - 1] = x11;
    tau[n - 2] = 0.0;
    tau[n - 1] = 0.0;
  }
  cluster_sync();
}

// A cluster per matrix: tridiagonalisation, then (want_k) the eigenpairs of the tridiagonal with
// eigenvalue >= thr, at most kmax: count by Sturm sequence, multisection, inverse iteration.
// The vectors go to the scratch (FP64, [k][n]), orthogonal up to the rounding of inverse iteration
// (k_eig_gram, k_eig_orth finish them).
//
// Eigenvalues: multisection on FP64 Sturm counts (sturm_count_minors), spread over the CTAs.
// Inverse iteration: a vector per LANE (lane-interleaved factorisations in the scratch), groups of 32
// vectors spread over the CTAs: two solves from a seeded start, then one more.  A vector of an
// eigenvalue with a gap g to its neighbours keeps ~eps ||T|| / g of theirs.  Gaps below OR_TOL ||T||
// are treated as a cluster (Gram-Schmidt, one warp each); the rest, at most ~1e-9 in the overlaps, is
// removed for all vectors at once by one symmetric first-order step (k_eig_orth) whose own
// error is the square of that.  (Clusters at 1e-3 ||T|| as usual put most kept
// OSVs in one: at 760 virtuals and 317 kept, 90 of 470 ms were one warp's Gram-Schmidt.)
template <class R>
__global__ void __launch_bounds__(R::NTH, 1) k_eig_tri(double* T, int n, double thr, int kmax, double* wout, int* kout,
                                                      double* scratch, int* err, int cap, int nsw, int refl_df,
                                                      int want_k) {
  using E = typename R::E;
  extern __shared__ double dyn[];
  uint32_t rank, C;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
  const int b = blockIdx.x / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int npad = (n + 31) & ~31;
  double* A = T + (size_t)b * n * n;
  double* w = wout + (size_t)b * kmax;
  double* scr = scratch + (size_t)b * eig_osv_scratch_doubles(n, kmax);
  double* d = scr;
  double* e = scr + n;
  double* tau = scr + 2 * n;
  double* work = scr + 3 * n;
  E* s0 = reinterpret_cast<E*>(dyn);
  E* s1 = s0 + npad;
  E* s2 = s1 + npad;
  E* tiles = s2 + npad;
  E* stage = tiles + (size_t)cap * TD_TILE;
  tridiag_cluster<R>(A, n, d, e, tau, s0, s1, s2, tiles, cap, stage, nsw, reinterpret_cast<E*>(work), refl_df != 0,
                     (int)rank, (int)C);
  if (!want_k) return;
  __shared__ int s_k, s_nclu;
  __shared__ double s_lo, s_hi, s_norm, s_sc;
  double* ds = dyn;           // the tridiagonal scaled to ||T|| <= 1 by a power of two
  double* e2s = dyn + npad;
  if (warp == 0) {            // Gershgorin bounds and the scale
    double glo = 1e300, ghi = -1e300, nrm = 0.0;
    for (int t = lane; t < n; t += 32) {
      const double off = (t > 0 ? fabs(e[t - 1]) : 0.0) + (t + 1 < n ? fabs(e[t]) : 0.0);
      glo = fmin(glo, d[t] - off);
      ghi = fmax(ghi, d[t] + off);
      nrm = fmax(nrm, fabs(d[t]) + off);
    }
    glo = -warp_max(-glo);
    ghi = warp_max(ghi);
    nrm = warp_max(nrm);
    if (lane == 0) {
      int ex = 0;
      if (nrm > 0.0 && isfinite(nrm)) frexp(nrm, &ex);
      const double sc = ldexp(1.0, max(-1000, min(1000, -ex))), span = (ghi - glo) * sc;
      s_lo = glo * sc - 1e-14 * span - 1e-290;
      s_hi = ghi * sc + 1e-14 * span + 1e-290;
      s_norm = nrm;
      s_sc = sc;
    }
  }
  __syncthreads();
  const double sc = s_sc, norm = s_norm;
  for (int t = tid; t < n; t += R::NTH) {
    ds[t] = d[t] * sc;
    const double ev = t + 1 < n ? e[t] * sc : 0.0;
    e2s[t] = fmax(ev * ev, 1e-60);
  }
  __syncthreads();
  if (warp == 0) {
    const int above = n - sturm_count_minors(ds, e2s, n, thr * sc);
    if (lane == 0) {
      s_k = min(above, kmax);
      if (rank == 0) {
        if (above > kmax) atomicOr(err, ERR_SIZE);
        kout[b] = min(above, kmax);
      }
    }
  }
  __syncthreads();
  const int k = s_k, gw = (int)rank + (int)C * warp, tw = (int)C * (R::NTH / 32);
  if (R::DF) {   // every warp: the FP32 pipes take them all
    dfl* dd = reinterpret_cast<dfl*>(ds);
    dfl* de = reinterpret_cast<dfl*>(e2s);
    for (int t = tid; t < n; t += R::NTH) {
      dd[t] = df_from(ds[t]);
      de[t] = df_from(e2s[t]);
    }
    __syncthreads();
    multisect_eigs_df(dd, de, n, k, gw, tw, s_lo, s_hi, 1e-30f, 5.7e-14 * norm * sc, 1.0 / sc, w);
  } else {       // this CTA's t = rank, rank + C, ... on four warps (one per FP64 pipe) unless one lane each takes more
    const int kc = (k + (int)C - 1) / (int)C, wm = min(R::NTH / 32, max(4, (kc + 31) / 32));
    if (warp < wm)
      multisect_eigs(ds, e2s, n, k, gw, (int)C * wm, s_lo, s_hi, 4.0 * 2.220446049250313e-16 * norm * sc, 1.0 / sc, w);
  }
  cluster_sync();   // the eigenvalues of every warp; s0 .. s2 are free
  E* dv = s0;
  E* ev = s1;
  int* clu = reinterpret_cast<int*>(s2);     // n + 1 ints
  for (int t = tid; t < n; t += R::NTH) {
    dv[t] = R::from(d[t]);
    ev[t] = t + 1 < n ? R::from(e[t]) : R::zero();
  }
  if (tid == 0) {
    int nc = 0;
    bool bad = false;
    double prev = 0.0;
    for (int t = 0; t < k; t++) {
      const double x = w[t];
      bad |= !isfinite(x);
      if (t == 0 || prev - x > OR_TOL * norm) clu[nc++] = t;
      prev = x;
    }
    clu[nc] = k;
    s_nclu = nc;
    if (bad && rank == 0) atomicOr(err, ERR_NONFINITE);
  }
  __syncthreads();
  E* VE = reinterpret_cast<E*>(work + eig_osv_work_doubles(n));   // [k][n]
  const double small = 2.220446049250313e-16 * fmax(norm, 1e-300);
  // factorisation slots, at most one a warp: above order 16 x 176 the room holds more of them than one CTA has warps
  const int nslot = min((int)(eig_osv_work_doubles(n) / ((size_t)176 * n)), tw);   // >= 4
  const int slot = gw;
  for (int pass = 0; pass < 2; pass++) {
    if (slot < nslot) {
      double* base = work + (size_t)slot * 176 * n;
      E* ui = reinterpret_cast<E*>(base) + lane;
      E* u1 = reinterpret_cast<E*>(base + 32 * (size_t)n) + lane;
      E* u2 = reinterpret_cast<E*>(base + 64 * (size_t)n) + lane;
      E* mul = reinterpret_cast<E*>(base + 96 * (size_t)n) + lane;
      E* y = reinterpret_cast<E*>(base + 128 * (size_t)n) + lane;
      int* piv = reinterpret_cast<int*>(base + 160 * (size_t)n) + lane;
      for (int g = slot; 32 * g < k; g += nslot) {
        const int t = 32 * g + lane;
        if (t < k) {
          // the second pass reuses the first pass's factorisation when every group kept its slot
          if (pass == 0 || k > 32 * nslot) R::factor(dv, ev, n, w[t], small, ui, u1, u2, mul, piv);
          if (pass == 0) {
#pragma unroll 4
            for (int r = 0; r < n; r++) {
              const uint64_t h = draw(0x5eedull + (uint64_t)t, (uint64_t)r);
              y[32 * r] = R::from((double)(h >> 40) * 0x1p-24 - 0.5);
            }
          } else {
#pragma unroll 8
            for (int r = 0; r < n; r++) y[32 * r] = VE[(size_t)t * n + r];
          }
          double sc = 1.0;   // scale of the previous solve, applied on the next read
          for (int it = 0; it < 2 - pass; it++) sc = R::solve(n, sc, ui, u1, u2, mul, piv, y);
          const E s = R::from(sc);
#pragma unroll 8
          for (int r = 0; r < n; r++) VE[(size_t)t * n + r] = R::mul(s, y[32 * r]);
        }
      }
    }
    cluster_sync();
    for (int c = gw; c < s_nclu; c += tw) {   // Gram-Schmidt within clusters, normalisation
      const int t0 = clu[c], t1 = clu[c + 1];
      for (int t = t0; t < t1; t++) {
        E* Vt = VE + (size_t)t * n;
        for (int s = t0; s < t; s++) {
          const E* Vs = VE + (size_t)s * n;
          const E nd = R::neg(warp_dot<R>(Vt, Vs, n));
          for (int r = lane; r < n; r += 32) Vt[r] = R::fma1(nd, Vs[r], Vt[r]);
          __syncwarp();
        }
        const double nn = R::to(warp_dot<R>(Vt, Vt, n));
        const E sc = R::from(nn > 0.0 ? 1.0 / sqrt(nn) : 0.0);
        for (int r = lane; r < n; r += 32) Vt[r] = R::mul(Vt[r], sc);
        __syncwarp();
      }
    }
    cluster_sync();
  }
  if (R::DF) {   // the vectors to FP64, in place
    double* VD = reinterpret_cast<double*>(VE);
    for (size_t i = (size_t)rank * R::NTH + tid; i < (size_t)k * n; i += (size_t)C * R::NTH) VD[i] = R::to(VE[i]);
  }
}

// G = V V^T (k x k, to the work room) of the vectors in the scratch: one 64 x 64 tile (tr >= tc) per CTA.
struct VRows {
  const double* V;
  int n;
  __device__ __forceinline__ double get(int t, int r) const { return V[(size_t)t * n + r]; }
};
struct VCols {
  const double* V;
  int n;
  __device__ __forceinline__ double get(int r, int t) const { return V[(size_t)t * n + r]; }
};
__global__ void __launch_bounds__(NT) k_eig_gram(int n, int kmax, const int* kout, double* scratch) {
  __shared__ double sm[GEMM_SMEM_DOUBLES];
  const int b = blockIdx.x, k = kout[b];
  int t = blockIdx.y, tr = 0;
  while ((tr + 1) * (tr + 2) / 2 <= t) tr++;
  const int tc = t - tr * (tr + 1) / 2;
  if (tr * TM >= k) return;
  double* work = scratch + (size_t)b * eig_osv_scratch_doubles(n, kmax) + 3 * n;
  const double* V = work + eig_osv_work_doubles(n);
  double acc[4][4] = {};
  tile_mma(k, k, n, tr * TM, tc * TN, VRows{V, n}, VCols{V, n}, acc, sm);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int u = 0; u < 4; u++)
#pragma unroll
    for (int v = 0; v < 4; v++) {
      const int r = tr * TM + ty + 16 * u, c = tc * TN + tx + 16 * v;
      if (r < k && c < k) {
        work[(size_t)r * k + c] = acc[u][v];
        work[(size_t)c * k + r] = acc[u][v];
      }
    }
}
// V <- V - (G - I) V / 2: the first-order symmetric orthogonalisation, into the output [k][n].
// Against Gram-Schmidt this is two products of k x k x n on the whole GPU.
struct GOff {
  const double* G;
  int k;
  __device__ __forceinline__ double get(int t, int q) const { return G[(size_t)t * k + q] - (t == q ? 1.0 : 0.0); }
};
__global__ void __launch_bounds__(NT) k_eig_orth(int n, int kmax, const int* kout, const double* scratch, double* Vout) {
  __shared__ double sm[GEMM_SMEM_DOUBLES];
  const int b = blockIdx.x, k = kout[b];
  const int nt = (n + TN - 1) / TN, tr = blockIdx.y / nt, tc = blockIdx.y % nt;
  if (tr * TM >= k) return;
  const double* work = scratch + (size_t)b * eig_osv_scratch_doubles(n, kmax) + 3 * n;
  const double* V = work + eig_osv_work_doubles(n);
  double* Vb = Vout + (size_t)b * n * kmax;
  double acc[4][4] = {};
  tile_mma(k, n, k, tr * TM, tc * TN, GOff{work, k}, VRows{V, n}, acc, sm);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int u = 0; u < 4; u++)
#pragma unroll
    for (int v = 0; v < 4; v++) {
      const int r = tr * TM + ty + 16 * u, c = tc * TN + tx + 16 * v;
      if (r < k && c < n) Vb[(size_t)r * n + c] = V[(size_t)r * n + c] - 0.5 * acc[u][v];
    }
}

// Shared memory of k_eig_tri with C CTAs per matrix: resident tiles and sweeping warps.
void td_layout(int n, int C, int nws, int* cap, int* nsw) {
  const size_t npad = (n + 31) & ~31, nb = npad / 32, nt = nb * (nb + 1) / 2, per = (nt + C - 1) / C;
  const size_t room = TD_SMEM / sizeof(double) > 3 * npad ? TD_SMEM / sizeof(double) - 3 * npad : 0;
  if (per * TD_TILE <= room) {
    *cap = (int)per;
    *nsw = nws;
    return;
  }
  *nsw = (int)std::min<size_t>(nws, room / TD_STAGE);
  *cap = (int)((room - (size_t)*nsw * TD_STAGE) / TD_TILE);
}
size_t td_smem(int n, int C, int nws) {
  int cap, nsw;
  td_layout(n, C, nws, &cap, &nsw);
  const size_t npad = (n + 31) & ~31;
  const size_t full = ((size_t)(npad / 32) * (npad / 32 + 1) / 2 + C - 1) / C;
  return (3 * npad + (size_t)cap * TD_TILE + (full <= (size_t)cap ? 0 : (size_t)nsw * TD_STAGE)) * sizeof(double);
}

// CTAs per matrix, measured at order 243 / 48 matrices: 1 CTA 7.6 ms, 2 5.3, 3 (46 clusters fit: two
// passes) 8.2; order 40 / 6: 1 CTA 0.59, 4 0.54, 8 0.51; order 640 / 128, double-float: 1 CTA 42, 2 49.
// The least of passes x (n steps of fixed latency + the sweep's share), passes = matrices /
// clusters that fit the GPU at a time (nclu[C], asked of the runtime once per context).
int eig_cluster_size(int n, int nb, bool df, const int* nclu) {
  const double lat1 = 5.5e-6, latc = 6e-6, tile = df ? 0.9e-6 : 1.1e-6;   // seconds per step, per tile sweep
  double tiles = 0.0;
  for (int L = 1; L < n; L++) {
    const double q = (L + 31) / 32;
    tiles += q * (q + 1) / 2;
  }
  int best = 1;
  double tb = 0.0;
  for (int C = 1; C <= 8; C++) {
    if (nclu[C] <= 0) continue;
    const double passes = (nb + nclu[C] - 1) / nclu[C];
    const double t = passes * (n * (C == 1 ? lat1 : latc) + tiles * tile / C);
    if (C == 1 || t < 0.97 * tb) {
      best = C;
      tb = t;
    }
  }
  return best;
}

template <class R>
void launch_tri(double* T, int nb, int n, double thr, int kmax, double* w, int* k, double* scratch, int* err, int C,
                int refl_df, int want_k, cudaStream_t st) {
  int cap, nsw;
  td_layout(n, C, R::NWS, &cap, &nsw);
  const size_t smem = td_smem(n, C, R::NWS);
  cudaFuncSetAttribute(k_eig_tri<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TD_SMEM);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nb * C);
  cfg.blockDim = dim3(R::NTH);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_eig_tri<R>, T, n, thr, kmax, w, k, scratch, err, cap, nsw, refl_df, want_k);
  note_launch(1);
}

}  // namespace

bool eig_order_fits(int n) {
  int cap, nsw;
  td_layout(n, 8, ArD::NWS, &cap, &nsw);
  return nsw > 0;
}

void eig_cluster_table(int* nclu) {
  cudaFuncSetAttribute(k_eig_tri<ArD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TD_SMEM);
  for (int C = 1; C <= 8; C++) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(ArD::NTH);
    cfg.dynamicSmemBytes = TD_SMEM;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int m = 0;
    if (cudaOccupancyMaxActiveClusters(&m, k_eig_tri<ArD>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      m = 0;
    }
    nclu[C] = m;
  }
  if (nclu[1] <= 0) nclu[1] = 1;
}

void launch_eig_tridiag(double* T, int nb, int n, int kmax, double* scratch, int* err, const int* nclu,
                        cudaStream_t st) {
  const int C = eig_cluster_size(n, nb, false, nclu);
  launch_tri<ArD>(T, nb, n, 0.0, kmax, nullptr, nullptr, scratch, err, C, 0, 0, st);
}

void launch_eig_topk(double* T, int nb, int n, double thr, int kmax, double* V, double* w, int* k, double* scratch,
                     int* err, bool df, bool refl_df, const int* nclu, cudaStream_t st) {
  const int C = eig_cluster_size(n, nb, df, nclu);
  if (df) launch_tri<ArF>(T, nb, n, thr, kmax, w, k, scratch, err, C, refl_df, 1, st);
  else launch_tri<ArD>(T, nb, n, thr, kmax, w, k, scratch, err, C, 0, 1, st);
  const int mt = (std::min(kmax, n) + TM - 1) / TM, nt = (n + TN - 1) / TN;
  k_eig_gram<<<dim3(nb, mt * (mt + 1) / 2), NT, 0, st>>>(n, kmax, k, scratch);
  k_eig_orth<<<dim3(nb, mt * nt), NT, 0, st>>>(n, kmax, k, scratch, V);
  note_launch(2);
}

}  // namespace osv

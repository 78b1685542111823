// Shared device building blocks of libosvmp2: block-matrix views, a CTA-wide
// FP64 tiled GEMM, deterministic CTA reductions and the device form of the
// counter-based generator that regenerates the RI integrals B.
#pragma once
#include <type_traits>
#include <cuda_runtime.h>
#include <stdint.h>

namespace osv {

constexpr int NT = 256;          // threads of every CTA that calls the CTA routines
constexpr int TM = 64, TN = 64, TK = 16;
constexpr int GEMM_SMEM_DOUBLES = TK * (TM + TN);
constexpr int GEMM_SMEM_F32 = TK * 2 * 97;   // floats: the (padded) 96 x 96 tiles of cta_gemm_f32s

// ---------------------------------------------------------------- views
// One dense block: element (r,c) at p[r*ld + c], or at p[c*ld + r] when tr.
struct Blk {
  const double* p;
  int ld;
  int tr;
};

// A matrix of up to 2x2 dense blocks.  Rows [0,rs) use block row 0, rows
// [rs,rows) block row 1; columns likewise with cs.  This is exactly the shape
// of the 4-block OSV pair matrices A_(ij,kl) (Eq. 4block_osv).
struct View {
  int rows, cols, rs, cs;
  Blk b[2][2];
  __device__ __forceinline__ double get(int r, int c) const {
    const int br = r >= rs, bc = c >= cs;
    const Blk& B = b[br][bc];
    const int rr = br ? r - rs : r, cc = bc ? c - cs : c;
    return B.tr ? B.p[(size_t)cc * B.ld + rr] : B.p[(size_t)rr * B.ld + cc];
  }
};

__host__ __device__ inline View dense_view(const double* p, int rows, int cols, int ld, int tr = 0) {
  View v;
  v.rows = rows; v.cols = cols; v.rs = rows; v.cs = cols;
  for (int a = 0; a < 2; a++)
    for (int c = 0; c < 2; c++) v.b[a][c] = Blk{p, ld, tr};
  return v;
}

// Transpose of a view (no data movement).
__host__ __device__ inline View transpose(const View& v) {
  View t;
  t.rows = v.cols; t.cols = v.rows; t.rs = v.cs; t.cs = v.rs;
  for (int a = 0; a < 2; a++)
    for (int c = 0; c < 2; c++) {
      t.b[a][c] = v.b[c][a];
      t.b[a][c].tr ^= 1;
    }
  return t;
}

// ---------------------------------------------------------------- double-float
// Unevaluated sums hi + lo of two FP32 numbers (~48 significant bits), with the
// error-free transformations of Knuth (two-sum) and Dekker (fast two-sum) and
// the FMA-based exact product.  On this part FP32 runs at 64x the FP64 rate, so
// an FMA in this arithmetic (~16 FP32 operations) costs a quarter of an FP64 FMA.
struct dfl {
  float h, l;
};
__device__ __forceinline__ dfl df_from(double x) {
  const float h = (float)x;
  return dfl{h, (float)(x - (double)h)};
}
__device__ __forceinline__ double df_to(dfl a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ dfl df_fast2(float a, float b) {   // |a| >= |b|
  const float s = a + b;
  return dfl{s, b - (s - a)};
}
__device__ __forceinline__ dfl df_add(dfl a, dfl b) {
  const float s = a.h + b.h;
  const float bb = s - a.h;
  const float e = (a.h - (s - bb)) + (b.h - bb);
  return df_fast2(s, e + (a.l + b.l));
}
__device__ __forceinline__ dfl df_mul(dfl a, dfl b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  return df_fast2(p, e);
}
__device__ __forceinline__ dfl df_neg(dfl a) { return dfl{-a.h, -a.l}; }
__device__ __forceinline__ dfl df_fma(dfl a, dfl b, dfl c) { return df_add(df_mul(a, b), c); }   // a b + c
__device__ __forceinline__ dfl df_shfl_xor(dfl a, int o) {
  return dfl{__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
}
// ---------------------------------------------------------------- GEMM
// Accumulate one TM x TN output tile at (m0, n0) of A[MxK] * B[KxN] into acc,
// in the arithmetic of V (double, or float for the low-precision products);
// views may hold either type and are converted on load.
// Thread (ty, tx) = (tid/16, tid%16) owns rows m0+ty+16i and cols n0+tx+16j.
template <class V, class VA, class VB>
__device__ __forceinline__ void tile_mma_t(int M, int N, int K, int m0, int n0, const VA& A, const VB& B,
                                           V acc[4][4], V* sm) {
  V* As = sm;             // [TK][TM]
  V* Bs = sm + TK * TM;   // [TK][TN]
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  // FP64: rows and columns of 16 past the end are skipped (an FMA holds the pipe for 64 cycles a warp)
  const int mi = sizeof(V) == 8 ? (min(M - m0, TM) + 15) / 16 : 4, nj = sizeof(V) == 8 ? (min(N - n0, TN) + 15) / 16 : 4;
  for (int k0 = 0; k0 < K; k0 += TK) {
#pragma unroll
    for (int t = 0; t < TM * TK / NT; t++) {
      const int e = tid + t * NT, m = e % TM, k = e / TM;
      const int gm = m0 + m, gk = k0 + k;
      As[k * TM + m] = (gm < M && gk < K) ? static_cast<V>(A.get(gm, gk)) : V(0);
    }
#pragma unroll
    for (int t = 0; t < TN * TK / NT; t++) {
      const int e = tid + t * NT, n = e % TN, k = e / TN;
      const int gn = n0 + n, gk = k0 + k;
      Bs[k * TN + n] = (gn < N && gk < K) ? static_cast<V>(B.get(gk, gn)) : V(0);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < TK; k++) {
      V a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; i++) a[i] = As[k * TM + ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; j++) b[j] = Bs[k * TN + tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; i++)
        if (sizeof(V) == 4 || i < mi) {
#pragma unroll
          for (int j = 0; j < 4; j++)
            if (sizeof(V) == 4 || j < nj) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
    }
    __syncthreads();
  }
}

// Error-free FP32 sum: s + e == a + b exactly (Knuth's two-sum).
__device__ __forceinline__ void two_sum_f(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// a + x1 y1 + x2 y2 in double-float arithmetic, the products' error terms gathered
// before one renormalisation (the rank-2 update of the tridiagonalisation sweep).
__device__ __forceinline__ dfl df_fma2(dfl x1, dfl y1, dfl x2, dfl y2, dfl a) {
  const float p1 = x1.h * y1.h;
  float e1 = fmaf(x1.h, y1.h, -p1);
  e1 = fmaf(x1.h, y1.l, e1);
  e1 = fmaf(x1.l, y1.h, e1);
  const float p2 = x2.h * y2.h;
  float e2 = fmaf(x2.h, y2.h, -p2);
  e2 = fmaf(x2.h, y2.l, e2);
  e2 = fmaf(x2.l, y2.h, e2);
  float s1, t1, s2, t2;
  two_sum_f(a.h, p1, s1, t1);
  two_sum_f(s1, p2, s2, t2);
  return df_fast2(s2, ((a.l + e1) + e2) + (t1 + t2));
}
// (h, l) += x y with (h, l) kept unnormalised: the leading sum by an exact two-sum,
// the error terms gathered in l (renormalised once by df_norm).
__device__ __forceinline__ void df_acc(float& h, float& l, dfl x, dfl y) {
  const float p = x.h * y.h;
  float e = fmaf(x.h, y.h, -p);
  e = fmaf(x.h, y.l, e);
  e = fmaf(x.l, y.h, e);
  float s, t;
  two_sum_f(h, p, s, t);
  h = s;
  l += e + t;
}
__device__ __forceinline__ dfl df_norm(float h, float l) {
  float s, e;
  two_sum_f(h, l, s, e);
  return dfl{s, e};
}
// a + x y in double-float arithmetic with one renormalisation (df_fma renormalises twice).
__device__ __forceinline__ dfl df_fma1(dfl x, dfl y, dfl a) {
  const float p = x.h * y.h;
  float e = fmaf(x.h, y.h, -p);
  e = fmaf(x.h, y.l, e);
  e = fmaf(x.l, y.h, e);
  float s, t;
  two_sum_f(a.h, p, s, t);
  return df_fast2(s, (a.l + e) + t);
}

// FP32 tile of (16 R) x (16 R) outputs, R x R per thread (thread (ty, tx) owns
// rows m0 + ty + 16 i and columns n0 + tx + 16 j), accumulated in FP32 over
// the whole K: for the short contractions (K ~ a pair order) of the coupling
// terms, whose FP32 rounding is scaled down by the off-diagonal Fock
// elements.  Each operand's k-tile is read along its contiguous direction
// (views report it through row_major()), and the next k-tile is loaded into
// registers while the current one is multiplied.  sm: 2 TK (16R + 1) floats.
template <int R, class VA, class VB>
__device__ __forceinline__ void tile_mma_f32r(int M, int N, int K, int m0, int n0, const VA& A, const VB& B,
                                              float acc[R][R], float* sm) {
  constexpr int TMR = 16 * R, LDT = TMR + 1, LPT = TMR * TK / NT;
  float* As = sm;             // [TK][LDT]
  float* Bs = sm + TK * LDT;  // [TK][LDT]
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const bool a_kf = A.row_major();   // A(m, k), A(m, k + 1) adjacent: walk k fastest
  const bool b_kf = !B.row_major();  // B(k, n), B(k + 1, n) adjacent: walk k fastest
  float ra[LPT], rb[LPT];
  auto load = [&](int k0) {
#pragma unroll
    for (int t = 0; t < LPT; t++) {
      const int e = tid + t * NT;
      const int m = a_kf ? e / TK : e % TMR, k = a_kf ? e % TK : e / TMR;
      const int gm = m0 + m, gk = k0 + k;
      ra[t] = (gm < M && gk < K) ? static_cast<float>(A.get(gm, gk)) : 0.f;
    }
#pragma unroll
    for (int t = 0; t < LPT; t++) {
      const int e = tid + t * NT;
      const int n = b_kf ? e / TK : e % TMR, k = b_kf ? e % TK : e / TMR;
      const int gn = n0 + n, gk = k0 + k;
      rb[t] = (gn < N && gk < K) ? static_cast<float>(B.get(gk, gn)) : 0.f;
    }
  };
  load(0);
  for (int k0 = 0; k0 < K; k0 += TK) {
#pragma unroll
    for (int t = 0; t < LPT; t++) {
      const int e = tid + t * NT;
      const int m = a_kf ? e / TK : e % TMR, k = a_kf ? e % TK : e / TMR;
      As[k * LDT + m] = ra[t];
      const int n = b_kf ? e / TK : e % TMR, kb = b_kf ? e % TK : e / TMR;
      Bs[kb * LDT + n] = rb[t];
    }
    __syncthreads();
    if (k0 + TK < K) load(k0 + TK);   // in flight during the products below
#pragma unroll
    for (int k = 0; k < TK; k++) {
      float a[R], b[R];
#pragma unroll
      for (int i = 0; i < R; i++) a[i] = As[k * LDT + ty + 16 * i];
#pragma unroll
      for (int j = 0; j < R; j++) b[j] = Bs[k * LDT + tx + 16 * j];
#pragma unroll
      for (int i = 0; i < R; i++)
#pragma unroll
        for (int j = 0; j < R; j++) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
}

template <int R, class CT, class VA, class VB>
__device__ void cta_gemm_f32r(int M, int N, int K, double alpha, const VA& A, const VB& B, double beta, CT* C, int ldc,
                              float* sm) {
  constexpr int TMR = 16 * R;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int m0 = 0; m0 < M; m0 += TMR)
    for (int n0 = 0; n0 < N; n0 += TMR) {
      float acc[R][R];
#pragma unroll
      for (int i = 0; i < R; i++)
#pragma unroll
        for (int j = 0; j < R; j++) acc[i][j] = 0.f;
      tile_mma_f32r<R>(M, N, K, m0, n0, A, B, acc, sm);
#pragma unroll
      for (int i = 0; i < R; i++)
#pragma unroll
        for (int j = 0; j < R; j++) {
          const int r = m0 + ty + 16 * i, c = n0 + tx + 16 * j;
          if (r < M && c < N) {
            CT* cp = C + (size_t)r * ldc + c;
            if constexpr (std::is_same<CT, float>::value)   // FP32 output: no FP64 work in the epilogue
              *cp = (beta == 0.0 ? 0.f : (float)beta * *cp) + (float)alpha * acc[i][j];
            else
              *cp = static_cast<CT>((beta == 0.0 ? 0.0 : beta * static_cast<double>(*cp)) + alpha * (double)acc[i][j]);
          }
        }
    }
  __syncthreads();
}

// (Chi, Clo) += alpha A B for short K in FP32 (tile_mma_f32r), each product
// folded into the compensated pair (Chi, Clo) with a two-sum: accumulation
// across many calls without FP64 arithmetic.
template <int R, class VA, class VB>
__device__ void cta_gemm_f32r_acc2(int M, int N, int K, float alpha, const VA& A, const VB& B, float* Chi, float* Clo,
                                   int ldc, float* sm) {
  constexpr int TMR = 16 * R;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int m0 = 0; m0 < M; m0 += TMR)
    for (int n0 = 0; n0 < N; n0 += TMR) {
      float acc[R][R];
#pragma unroll
      for (int i = 0; i < R; i++)
#pragma unroll
        for (int j = 0; j < R; j++) acc[i][j] = 0.f;
      tile_mma_f32r<R>(M, N, K, m0, n0, A, B, acc, sm);
#pragma unroll
      for (int i = 0; i < R; i++)
#pragma unroll
        for (int j = 0; j < R; j++) {
          const int r = m0 + ty + 16 * i, c = n0 + tx + 16 * j;
          if (r < M && c < N) {
            const size_t o = (size_t)r * ldc + c;
            float s, e;
            two_sum_f(Chi[o], alpha * acc[i][j], s, e);
            Chi[o] = s;
            Clo[o] += e;
          }
        }
    }
  __syncthreads();
}
// Tile set of the short FP32 contractions: 0 = 64 x 64 tiles up to 64 x 64
// outputs and 96 x 96 above; 1 = also 80 x 80 tiles for outputs up to 80 x 80.
// (A runtime choice of the solver's autotuner; the K order of every output's
// FMAs, hence the result, is the same for every tile shape.)
template <class VA, class VB>
__device__ void cta_gemm_f32s_acc2(int M, int N, int K, float alpha, const VA& A, const VB& B, float* Chi, float* Clo,
                                   int ldc, float* sm, int tiles = 0) {
  const int mx = max(M, N);
  if (mx <= TM)
    cta_gemm_f32r_acc2<4>(M, N, K, alpha, A, B, Chi, Clo, ldc, sm);
  else if (tiles == 1 && mx <= 80)
    cta_gemm_f32r_acc2<5>(M, N, K, alpha, A, B, Chi, Clo, ldc, sm);
  else
    cta_gemm_f32r_acc2<6>(M, N, K, alpha, A, B, Chi, Clo, ldc, sm);
}

// C = beta C + alpha A B for short K (<= a few hundred) in FP32 (tile_mma_f32r),
// 64 x 64 tiles for outputs up to 64 x 64 and 96 x 96 tiles (one pass over
// the usual pair orders ~80) above; sm holds GEMM_SMEM_F32 floats.
template <class CT, class VA, class VB>
__device__ void cta_gemm_f32s(int M, int N, int K, double alpha, const VA& A, const VB& B, double beta, CT* C, int ldc,
                              float* sm, int tiles = 0) {
  const int mx = max(M, N);
  if (mx <= TM)
    cta_gemm_f32r<4>(M, N, K, alpha, A, B, beta, C, ldc, sm);
  else if (tiles == 1 && mx <= 80)
    cta_gemm_f32r<5>(M, N, K, alpha, A, B, beta, C, ldc, sm);
  else
    cta_gemm_f32r<6>(M, N, K, alpha, A, B, beta, C, ldc, sm);
}


template <class VA, class VB>
__device__ __forceinline__ void tile_mma(int M, int N, int K, int m0, int n0, const VA& A, const VB& B,
                                         double acc[4][4], double* sm) {
  tile_mma_t<double>(M, N, K, m0, n0, A, B, acc, sm);
}

// C[MxN] (row-major, ldc, element type CT) = beta*C + alpha*A*B with the whole
// CTA (NT threads), products in the arithmetic of V.  beta == 0 never reads C.
template <class V, class CT, class VA, class VB>
__device__ void cta_gemm_t(int M, int N, int K, V alpha, const VA& A, const VB& B, V beta, CT* C, int ldc, V* sm) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int m0 = 0; m0 < M; m0 += TM)
    for (int n0 = 0; n0 < N; n0 += TN) {
      V acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = V(0);
      tile_mma_t<V>(M, N, K, m0, n0, A, B, acc, sm);
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
          const int r = m0 + ty + 16 * i, c = n0 + tx + 16 * j;
          if (r < M && c < N) {
            CT* cp = C + (size_t)r * ldc + c;
            *cp = static_cast<CT>((beta == V(0) ? V(0) : beta * static_cast<V>(*cp)) + alpha * acc[i][j]);
          }
        }
    }
  __syncthreads();
}

template <class VA, class VB>
__device__ void cta_gemm(int M, int N, int K, double alpha, const VA& A, const VB& B, double beta, double* C,
                         int ldc, double* sm) {
  cta_gemm_t<double, double>(M, N, K, alpha, A, B, beta, C, ldc, sm);
}

// FP64 GEMM with (16 R) x (16 R) output tiles, R x R per thread (thread (ty, tx)
// owns rows m0 + ty + 16 i and columns n0 + tx + 16 j); the K order of every
// output's FMAs is that of cta_gemm, so the results are the same.  sm: 2 TK 16R.
template <int R, class VA, class VB>
__device__ void cta_gemm_r(int M, int N, int K, double alpha, const VA& A, const VB& B, double beta, double* C,
                           int ldc, double* sm) {
  constexpr int TMR = 16 * R;
  double* As = sm;
  double* Bs = sm + TK * TMR;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int m0 = 0; m0 < M; m0 += TMR)
    for (int n0 = 0; n0 < N; n0 += TMR) {
      const int mi = (min(M - m0, TMR) + 15) / 16, nj = (min(N - n0, TMR) + 15) / 16;   // 16s with elements
      double acc[R][R];
#pragma unroll
      for (int i = 0; i < R; i++)
#pragma unroll
        for (int j = 0; j < R; j++) acc[i][j] = 0.0;
      for (int k0 = 0; k0 < K; k0 += TK) {
#pragma unroll
        for (int t = 0; t < TMR * TK / NT; t++) {
          const int e = tid + t * NT, m = e % TMR, k = e / TMR;
          const int gm = m0 + m, gk = k0 + k;
          As[k * TMR + m] = (gm < M && gk < K) ? static_cast<double>(A.get(gm, gk)) : 0.0;
        }
#pragma unroll
        for (int t = 0; t < TMR * TK / NT; t++) {
          const int e = tid + t * NT, n = e % TMR, k = e / TMR;
          const int gn = n0 + n, gk = k0 + k;
          Bs[k * TMR + n] = (gn < N && gk < K) ? static_cast<double>(B.get(gk, gn)) : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < TK; k++) {
          double a[R], b[R];
#pragma unroll
          for (int i = 0; i < R; i++) a[i] = As[k * TMR + ty + 16 * i];
#pragma unroll
          for (int j = 0; j < R; j++) b[j] = Bs[k * TMR + tx + 16 * j];
#pragma unroll
          for (int i = 0; i < R; i++)
            if (i < mi) {
#pragma unroll
              for (int j = 0; j < R; j++)
                if (j < nj) acc[i][j] = fma(a[i], b[j], acc[i][j]);
            }
        }
        __syncthreads();
      }
#pragma unroll
      for (int i = 0; i < R; i++)
#pragma unroll
        for (int j = 0; j < R; j++) {
          const int r = m0 + ty + 16 * i, c = n0 + tx + 16 * j;
          if (r < M && c < N) {
            double* cp = C + (size_t)r * ldc + c;
            *cp = (beta == 0.0 ? 0.0 : beta * *cp) + alpha * acc[i][j];
          }
        }
    }
  __syncthreads();
}

// cta_gemm with 96 x 96 tiles where they pad less than 64 x 64 ones (pair
// orders 65..96 fit one tile instead of four); sm holds GEMM_SMEM_WIDE doubles.
constexpr int GEMM_SMEM_WIDE = TK * 2 * 96;
template <class VA, class VB>
__device__ void cta_gemm_a(int M, int N, int K, double alpha, const VA& A, const VB& B, double beta, double* C,
                           int ldc, double* sm) {
  const long long p64 = (long long)((M + 63) / 64) * ((N + 63) / 64) * 4096;
  const long long p96 = (long long)((M + 95) / 96) * ((N + 95) / 96) * 9216;
  if (p96 < p64)
    cta_gemm_r<6>(M, N, K, alpha, A, B, beta, C, ldc, sm);
  else
    cta_gemm_r<4>(M, N, K, alpha, A, B, beta, C, ldc, sm);
}


// C = beta C + alpha A B in double-float arithmetic (FP32 pipes, ~48 bits): the
// FP64 views are converted as their tiles are staged, the products accumulate
// as (hi, lo) pairs in the K order of cta_gemm, C is written in FP64.  For the
// mixed form's FP64-shaped products whose inputs carry fewer bits than that.
// Tiles (16 R) x (16 R), R x R per thread; sm: 2 TK 16R doubles.
template <int R, class VA, class VB>
__device__ void cta_gemm_df_r(int M, int N, int K, double alpha, const VA& A, const VB& B, double beta, double* C,
                              int ldc, double* sm) {
  constexpr int TMR = 16 * R;
  dfl* As = reinterpret_cast<dfl*>(sm);
  dfl* Bs = As + TK * TMR;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int m0 = 0; m0 < M; m0 += TMR)
    for (int n0 = 0; n0 < N; n0 += TMR) {
      dfl acc[R][R];
#pragma unroll
      for (int i = 0; i < R; i++)
#pragma unroll
        for (int j = 0; j < R; j++) acc[i][j] = dfl{0.f, 0.f};
      for (int k0 = 0; k0 < K; k0 += TK) {
#pragma unroll
        for (int t = 0; t < TMR * TK / NT; t++) {
          const int e = tid + t * NT, m = e % TMR, k = e / TMR;
          const int gm = m0 + m, gk = k0 + k;
          As[k * TMR + m] = (gm < M && gk < K) ? df_from(static_cast<double>(A.get(gm, gk))) : dfl{0.f, 0.f};
        }
#pragma unroll
        for (int t = 0; t < TMR * TK / NT; t++) {
          const int e = tid + t * NT, n = e % TMR, k = e / TMR;
          const int gn = n0 + n, gk = k0 + k;
          Bs[k * TMR + n] = (gn < N && gk < K) ? df_from(static_cast<double>(B.get(gk, gn))) : dfl{0.f, 0.f};
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < TK; k++) {
          dfl a[R], b[R];
#pragma unroll
          for (int i = 0; i < R; i++) a[i] = As[k * TMR + ty + 16 * i];
#pragma unroll
          for (int j = 0; j < R; j++) b[j] = Bs[k * TMR + tx + 16 * j];
#pragma unroll
          for (int i = 0; i < R; i++)
#pragma unroll
            for (int j = 0; j < R; j++) df_acc(acc[i][j].h, acc[i][j].l, a[i], b[j]);   // unnormalised
        }
        __syncthreads();
      }
#pragma unroll
      for (int i = 0; i < R; i++)
#pragma unroll
        for (int j = 0; j < R; j++) {
          const int r = m0 + ty + 16 * i, c = n0 + tx + 16 * j;
          if (r < M && c < N) {
            double* cp = C + (size_t)r * ldc + c;
            *cp = (beta == 0.0 ? 0.0 : beta * *cp) + alpha * df_to(acc[i][j]);
          }
        }
    }
  __syncthreads();
}
// cta_gemm_df_r with 96- or 64-wide tiles, whichever pads less (as cta_gemm_a);
// sm holds GEMM_SMEM_WIDE doubles.
template <class VA, class VB>
__device__ void cta_gemm_df(int M, int N, int K, double alpha, const VA& A, const VB& B, double beta, double* C,
                            int ldc, double* sm) {
  const long long p64 = (long long)((M + 63) / 64) * ((N + 63) / 64) * 4096;
  const long long p96 = (long long)((M + 95) / 96) * ((N + 95) / 96) * 9216;
  if (p96 < p64)
    cta_gemm_df_r<6>(M, N, K, alpha, A, B, beta, C, ldc, sm);
  else
    cta_gemm_df_r<4>(M, N, K, alpha, A, B, beta, C, ldc, sm);
}

// Dense float matrix view (element (r,c) at p[r*ld+c], or p[c*ld+r] when tr).
struct ViewF {
  const float* p;
  int ld;
  int tr;
  __device__ __forceinline__ float get(int r, int c) const {
    return tr ? p[(size_t)c * ld + r] : p[(size_t)r * ld + c];
  }
  __device__ __forceinline__ bool row_major() const { return !tr; }   // (r, c), (r, c + 1) adjacent
};

// ---------------------------------------------------------------- reductions
// Deterministic CTA sum / max (fixed shuffle tree, then fixed order over warps).
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
// red: >= 33 doubles of shared memory. Result returned to every thread.
__device__ inline double cta_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < nw; k++) s += red[k];
    red[32] = s;
  }
  __syncthreads();
  return red[32];
}
__device__ inline float cta_sum(float v, float* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
    for (int k = 0; k < nw; k++) s += red[k];
    red[32] = s;
  }
  __syncthreads();
  return red[32];
}
__device__ inline double cta_max(double v, double* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_max(v);
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = red[0];
    for (int k = 1; k < nw; k++) s = fmax(s, red[k]);
    red[32] = s;
  }
  __syncthreads();
  return red[32];
}

// ---------------------------------------------------------------- generator
// SplitMix64 output finaliser (Steele, Lea & Flood 2014) and the draws built on
// it; B[i,a,P] = env[i,a] * z with z the Irwin-Hall sum of twelve 16-bit fields
// of three consecutive draws, shifted and scaled exactly by 2^-16.
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__host__ __device__ __forceinline__ uint64_t draw(uint64_t key, uint64_t c) {
  return mix64(key + (c + 1ull) * 0x9E3779B97F4A7C15ull);
}
__device__ __forceinline__ double ih12(uint64_t key, uint64_t ctr) {
  int64_t s = 0;
#pragma unroll
  for (int t = 0; t < 3; t++) {
    const uint64_t h = draw(key, 3ull * ctr + (uint64_t)t);
    s += (int64_t)(h & 0xFFFFull) + (int64_t)((h >> 16) & 0xFFFFull) + (int64_t)((h >> 32) & 0xFFFFull) +
         (int64_t)(h >> 48);
  }
  return (double)(s - 393210) * 0x1p-16;
}

// Source of B: stored array, or regeneration from (key, env).
struct BSrc {
  const double* B;
  const double* env;
  uint64_t key;
  int n_vir, n_aux;
  __device__ __forceinline__ double get(int i, int a, int P) const {
    const size_t idx = ((size_t)i * n_vir + a) * n_aux + P;
    if (B) return B[idx];
    return env[(size_t)i * n_vir + a] * ih12(key, (uint64_t)idx);
  }
};

// Device-side error flag bits written by kernels (read by the host after sync).
enum : int { ERR_EIG = 1, ERR_NONFINITE = 2, ERR_NOCONV = 4, ERR_SIZE = 8, ERR_TIMEOUT = 16 };

}  // namespace osv

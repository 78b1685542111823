// Operands and launches of the FP64 tensor-core contraction (tc_oz.cuh).
#include "internal.h"
#include "oz_split.cuh"
#include "tc_oz.cuh"

namespace osv {

// Rows already contiguous in k (stored or generated B with k = aux, dense row-major matrices): one warp per
// (row, chunk), lanes along k in pairs.
struct OzSrcB {            // row a of slot u: B[i0 + u][a][.]
  BSrc src;
  int i0;
  __device__ __forceinline__ double get(int u, int r, int k) const { return src.get(i0 + u, r, k); }
};
struct OzSrcBT {           // row P of slot u: B[xs[u]][.][P]
  BSrc src;
  const int* xs;
  __device__ __forceinline__ double get(int u, int r, int k) const { return src.get(xs[u], k, r); }
};

template <int NS, class Src>
__global__ void __launch_bounds__(256) k_oz_rows(Src src, int rows, int K, int ld, size_t slice,
                                                 uint16_t* __restrict__ D, int* __restrict__ ex) {
  const int u = blockIdx.y, lane = threadIdx.x & 31;
  const int nch = (K + oz::CHUNK - 1) / oz::CHUNK;
  const long long w = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (w >= (long long)rows * nch) return;   // warp-uniform
  const int r = (int)(w / nch), c = (int)(w % nch), k0 = c * oz::CHUNK;
  double x[8];
#pragma unroll
  for (int v = 0; v < 8; v++) {
    const int k = k0 + 64 * (v >> 1) + 2 * lane + (v & 1);
    x[v] = k < K ? src.get(u, r, k) : 0.0;
  }
  const int e = oz::warp_slices<NS>(x, min(oz::CHUNK, K - k0), D + ((size_t)u * rows + r) * ld + k0, slice, lane);
  if (lane == 0) ex[((size_t)u * rows + r) * nch + c] = e;
}

// Rows strided in k (their index innermost): one CTA per 16 rows x one chunk, transposed through shared memory so
// that both the reads (rows innermost) and the digit writes (k innermost) are coalesced.
template <int NS, class Src>
__global__ void __launch_bounds__(256) k_oz_cols(Src src, int rows, int K, int ld, size_t slice,
                                                 uint16_t* __restrict__ D, int* __restrict__ ex) {
  __shared__ double tile[oz::CHUNK][17];
  const int u = blockIdx.z, r0 = blockIdx.x * 16, c = blockIdx.y, k0 = c * oz::CHUNK;
  const int nch = (K + oz::CHUNK - 1) / oz::CHUNK;
  for (int t = threadIdx.x; t < oz::CHUNK * 16; t += 256) {
    const int k = t >> 4, r = t & 15;
    tile[k][r] = (k0 + k < K && r0 + r < rows) ? src.get(u, r0 + r, k0 + k) : 0.0;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int dr = threadIdx.x >> 5; dr < 16 && r0 + dr < rows; dr += 8) {   // warp-uniform
    double x[8];
#pragma unroll
    for (int v = 0; v < 8; v++) x[v] = tile[64 * (v >> 1) + 2 * lane + (v & 1)][dr];
    const int r = r0 + dr;
    const int e = oz::warp_slices<NS>(x, min(oz::CHUNK, K - k0), D + ((size_t)u * rows + r) * ld + k0, slice, lane);
    if (lane == 0) ex[((size_t)u * rows + r) * nch + c] = e;
  }
}

// A list of dense matrices with the row index innermost ([K][rows], row stride ldm), optionally scaled by w[k];
// digits zero up to kpad.
template <int NS>
__global__ void __launch_bounds__(256) k_oz_mats(const OzMat* __restrict__ mats, const double* __restrict__ w,
                                                 int ld, size_t slice, uint16_t* __restrict__ D, int* __restrict__ ex) {
  __shared__ double tile[oz::CHUNK][17];
  const OzMat mt = mats[blockIdx.z];
  const int r0 = blockIdx.x * 16, c = blockIdx.y, k0 = c * oz::CHUNK, K = mt.K;
  if (r0 >= mt.rows || k0 >= K) return;
  for (int t = threadIdx.x; t < oz::CHUNK * 16; t += 256) {
    const int k = t >> 4, r = t & 15;
    double v = 0.0;
    if (k0 + k < K && r0 + r < mt.rows) {
      v = mt.p[(size_t)(k0 + k) * mt.ldm + r0 + r];
      if (w) v *= w[k0 + k];
    }
    tile[k][r] = v;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int dr = threadIdx.x >> 5; dr < 16 && r0 + dr < mt.rows; dr += 8) {
    double x[8];
#pragma unroll
    for (int v = 0; v < 8; v++) x[v] = tile[64 * (v >> 1) + 2 * lane + (v & 1)][dr];
    const int r = r0 + dr;
    const int e = oz::warp_slices<NS>(x, min(oz::CHUNK, mt.kpad - k0), D + ((size_t)mt.m.row + r) * ld + k0, slice, lane);
    if (lane == 0) ex[mt.m.eb + (size_t)r * mt.m.es + c] = e;
  }
}
// The same for matrices with k innermost ([rows][K], row stride ldm): a warp per (row, chunk).
template <int NS>
__global__ void __launch_bounds__(256) k_oz_rmats(const OzMat* __restrict__ mats, int ld, size_t slice,
                                                  uint16_t* __restrict__ D, int* __restrict__ ex) {
  const OzMat mt = mats[blockIdx.z];
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), c = blockIdx.y, k0 = c * oz::CHUNK, lane = threadIdx.x & 31;
  if (r >= mt.rows || k0 >= mt.K) return;
  double x[8];
#pragma unroll
  for (int v = 0; v < 8; v++) {
    const int k = k0 + 64 * (v >> 1) + 2 * lane + (v & 1);
    x[v] = k < mt.K ? mt.p[(size_t)r * mt.ldm + k] : 0.0;
  }
  const int e = oz::warp_slices<NS>(x, min(oz::CHUNK, mt.kpad - k0), D + ((size_t)mt.m.row + r) * ld + k0,
                                slice, lane);
  if (lane == 0) ex[mt.m.eb + (size_t)r * mt.m.es + c] = e;
}

// Matrices of FP32 pairs with k innermost (mixed form: G and its remainder, lo_shift floats further on): a warp per
// (row, chunk); the fixed-point numbers without the FP64 pipe, whose conversions would take longer than the reads.
template <int NS>
__global__ void __launch_bounds__(256) k_oz_pairs(const OzMat* __restrict__ mats, long long lo_shift, int ld, size_t slice,
                                                  uint16_t* __restrict__ D, int* __restrict__ ex) {
  constexpr int T = 7 + 8 * (NS - 1);                  // |x| < 2^e -> |F| < 2^T
  const OzMat mt = mats[blockIdx.z];
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), c = blockIdx.y, k0 = c * oz::CHUNK, lane = threadIdx.x & 31;
  if (r >= mt.rows || k0 >= mt.K) return;
  const float* g = reinterpret_cast<const float*>(mt.p) + (size_t)r * mt.ldm;
  float h[8], l[8];
  unsigned mx = 0;
#pragma unroll
  for (int v = 0; v < 8; v++) {
    const int k = k0 + 64 * (v >> 1) + 2 * lane + (v & 1);
    h[v] = k < mt.K ? g[k] : 0.f;
    l[v] = k < mt.K ? g[k + lo_shift] : 0.f;
    mx = max(mx, (unsigned)__float_as_int(h[v]) & 0x7fffffffu);
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  const int fe = (int)(mx >> 23);                      // below 2^-80: zero
  const int e = fe == 255 ? oz::EX_NAN : (fe < 47 ? oz::EX_ZERO : fe - 126);
  const bool live = fe != 255 && fe >= 47;
  const int sh = live ? T - 16 - e : 0;                // |h 2^sh| < 2^(T - 16) <= 2^23
  const float s0 = __int_as_float(((sh >> 1) + 127) << 23), s1 = __int_as_float((sh - (sh >> 1) + 127) << 23);
  uint16_t* dst = D + ((size_t)mt.m.row + r) * ld + k0;
  const int kv = min(oz::CHUNK, mt.kpad - k0);
#pragma unroll
  for (int u = 0; u < 4; u++) {
    const int k = 64 * u + 2 * lane;
    if (k >= kv) continue;
    long long f[2];
#pragma unroll
    for (int w = 0; w < 2; w++) {
      const float a = live ? h[2 * u + w] * s0 * s1 : 0.f, b = live ? l[2 * u + w] * s0 * s1 : 0.f;
      const int top = __float2int_rn(a);
      f[w] = ((long long)top << 16) + __float2int_rn(fmaf(a - (float)top, 65536.f, b * 65536.f));
    }
#pragma unroll
    for (int s = NS - 1; s >= 0; s--) *reinterpret_cast<uint32_t*>(dst + s * slice + k) = oz::digit_pair(f[0], f[1], s);
  }
  if (lane == 0) ex[mt.m.eb + (size_t)r * mt.m.es + c] = e;
}
__global__ void k_oz_float(const double* __restrict__ x, size_t n, float* __restrict__ y) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) y[i] = (float)x[i];
}

// One call of f<NS> for the slice counts in use.
#define OZ_DISPATCH(ns, call)                                  \
  do {                                                         \
    if ((ns) == oz::NSL) { constexpr int NS = oz::NSL; call; } \
    else { constexpr int NS = oz::MXSL; call; }                \
  } while (0)

void launch_oz_rows(const BSrc& src, int i0, int nb, int ns, uint16_t* D, int* ex, cudaStream_t st) {
  if (!nb) return;
  const size_t slice = (size_t)nb * src.n_vir * oz::ld_of(src.n_aux);
  const long long warps = (long long)src.n_vir * oz::n_chunks(src.n_aux);
  const dim3 grid((unsigned)((warps + 7) / 8), nb);
  OZ_DISPATCH(ns, (k_oz_rows<NS><<<grid, 256, 0, st>>>(OzSrcB{src, i0}, src.n_vir, src.n_aux, oz::ld_of(src.n_aux), slice, D, ex)));
  note_launch(1);
}
void launch_oz_cols(const BSrc& src, const int* xs, int nb, int ns, uint16_t* D, int* ex, cudaStream_t st) {
  if (!nb) return;
  const size_t slice = (size_t)nb * src.n_aux * oz::ld_of(src.n_vir);
  const dim3 grid((src.n_aux + 15) / 16, oz::n_chunks(src.n_vir), nb);
  OZ_DISPATCH(ns, (k_oz_cols<NS><<<grid, 256, 0, st>>>(OzSrcBT{src, xs}, src.n_aux, src.n_vir, oz::ld_of(src.n_vir), slice, D, ex)));
  note_launch(1);
}
void launch_oz_mats(const OzMat* mats, int n, int max_rows, int max_K, const double* w, bool k_inner, int ns, int ld,
                    long long rows, uint16_t* D, int* ex, cudaStream_t st) {
  if (!n) return;
  const size_t slice = (size_t)rows * ld;
  for (int q = 0; q < n; q += 65535) {     // grid z limit
    const int nq = n - q < 65535 ? n - q : 65535;
    const dim3 gr((max_rows + 7) / 8, oz::n_chunks(max_K), nq), gc((max_rows + 15) / 16, oz::n_chunks(max_K), nq);
    if (k_inner) OZ_DISPATCH(ns, (k_oz_rmats<NS><<<gr, 256, 0, st>>>(mats + q, ld, slice, D, ex)));
    else OZ_DISPATCH(ns, (k_oz_mats<NS><<<gc, 256, 0, st>>>(mats + q, w, ld, slice, D, ex)));
    note_launch(1);
  }
}

void launch_mx_pairs(const OzMat* mats, int n, int max_rows, int K, long long lo_shift, int ld, long long rows, uint16_t* D,
                     int* ex, cudaStream_t st) {
  for (int q = 0; q < n; q += 65535) {     // grid z limit
    const int nq = n - q < 65535 ? n - q : 65535;
    k_oz_pairs<oz::MXSL><<<dim3((max_rows + 7) / 8, oz::n_chunks(K), nq), 256, 0, st>>>(mats + q, lo_shift, ld, (size_t)rows * ld, D, ex);
    note_launch(1);
  }
}
void launch_oz_float(const double* x, size_t n, float* y, cudaStream_t st) {
  if (!n) return;
  k_oz_float<<<1184, 256, 0, st>>>(x, n, y);
  note_launch(1);
}

// out[row][col] (row-major), added to what is there when job.s = 1
struct OzEpiRow {
  static constexpr bool kWarp = false, kDigits = false, kPair = false, kLong = false;
  __device__ __forceinline__ void operator()(const oz::Job& jb, int r, int c0, const double (&v)[oz::DCOL]) const {
    double* o = static_cast<double*>(jb.out) + (size_t)(jb.m0 + r) * jb.ld_out + jb.n0 + c0;
#pragma unroll
    for (int u = 0; u < oz::DCOL; u++)
      if (c0 + u < jb.n_valid) o[u] = jb.s == 0.0 ? v[u] : o[u] + v[u];
  }
};
// Mixed form.  G = U^T B with the row (aux) index innermost, as a normalised FP32 pair: the leading part to
// out[col][row], the remainder lo_shift floats further on.
struct OzEpiG {
  static constexpr bool kWarp = false, kDigits = false, kPair = true, kLong = false;
  long long lo_shift;
  __device__ __forceinline__ void pairs(const oz::Job& jb, int r, int c0, const float (&h)[oz::DCOL],
                                        const float (&l)[oz::DCOL]) const {
    float* o = static_cast<float*>(jb.out) + (size_t)(jb.n0 + c0) * jb.ld_out + jb.m0 + r;
#pragma unroll
    for (int u = 0; u < oz::DCOL; u++)
      if (c0 + u < jb.n_valid) {
        const dfl v = df_norm(h[u], l[u]);
        o[(size_t)u * jb.ld_out] = v.h;
        o[(size_t)u * jb.ld_out + lo_shift] = v.l;
      }
  }
};
// out[row][col], FP64 (K~) or FP32 (Sigma)
template <class T>
struct OzEpiPair {
  static constexpr bool kWarp = false, kDigits = false, kPair = true, kLong = false;
  __device__ __forceinline__ void pairs(const oz::Job& jb, int r, int c0, const float (&h)[oz::DCOL],
                                        const float (&l)[oz::DCOL]) const {
    T* o = static_cast<T*>(jb.out) + (size_t)(jb.m0 + r) * jb.ld_out + jb.n0 + c0;
#pragma unroll
    for (int u = 0; u < oz::DCOL; u++)
      if (c0 + u < jb.n_valid) o[u] = (T)h[u] + (T)l[u];
  }
};
// T[a][b] = T[b][a] = v / (e_a + e_b - s) for a >= b; out = T_i, s = 2 f_ii
struct OzEpiT {
  static constexpr bool kWarp = false, kDigits = false, kPair = false, kLong = false;
  const double* e_vir;
  __device__ __forceinline__ void operator()(const oz::Job& jb, int r, int c0, const double (&v)[oz::DCOL]) const {
    const int a = jb.m0 + r;
    const double ea = e_vir[a] - jb.s;
    double* T = static_cast<double*>(jb.out);
#pragma unroll
    for (int u = 0; u < oz::DCOL; u++) {
      const int b = jb.n0 + c0 + u;
      if (c0 + u < jb.n_valid && a >= b) {
        const double t = v[u] / (ea + e_vir[b]);
        T[(size_t)a * jb.ld_out + b] = t;
        T[(size_t)b * jb.ld_out + a] = t;
      }
    }
  }
};

// Mixed amplitude iterations.  Sigma has the exponent 1 (|x| <= 1 + rounding), Y and W one exponent a matrix.
// W: the digits of c Sigma op(Y)^T under the exponent code eP[o_e] of its pair; c = job.s, Y's code eY[job.ld_out].
struct OzEpiW {
  static constexpr bool kWarp = false, kDigits = false, kPair = true, kLong = true;
  static constexpr int NS = oz::MXSOLVE, T = 7 + 8 * (NS - 1);
  uint16_t* D;
  int ld;
  size_t slice;
  const int *eY, *eP;
  struct Scale {
    float ch, cl;          // c 2^(exponents) as a pair: the fixed-point number per unit of the first level
  };
  __device__ __forceinline__ Scale scale(const oz::Job& jb) const {
    const int ey = eY[jb.ld_out], ep = eP[jb.o_e];
    if (ey < oz::EX_ZERO / 2 || ep < oz::EX_ZERO / 2 || ey > oz::EX_NAN / 2 || ep > oz::EX_NAN / 2) return Scale{0.f, 0.f};
    const int x = T - ep + 1 + ey - 14;                // |c v| 2^x < 2^T
    const float h = (float)jb.s, l = (float)(jb.s - (double)h);
    const float s0 = __int_as_float(((x >> 1) + 127) << 23), s1 = __int_as_float((x - (x >> 1) + 127) << 23);
    return Scale{h * s0 * s1, l * s0 * s1};
  }
  __device__ __forceinline__ void tile(const oz::Job& jb, const Scale& sc, int r, int c0, const float (&vh)[oz::DCOL],
                                       const float (&vl)[oz::DCOL]) const {
    uint16_t* o = D + ((size_t)jb.o_row + jb.m0 + r) * ld + jb.n0 + c0;
    const bool tail = c0 + oz::DCOL >= jb.n_valid && ((jb.n0 + c0) & 16) == 0;   // also clears the rest of a k-block
    int f[oz::DCOL];
#pragma unroll
    for (int u = 0; u < oz::DCOL; u++) {
      const float p = vh[u] * sc.ch;
      float e = fmaf(vh[u], sc.ch, -p);
      e = fmaf(vh[u], sc.cl, e);
      e = fmaf(vl[u], sc.ch, e);
      const int top = __float2int_rn(p);
      f[u] = c0 + u < jb.n_valid ? top + __float2int_rn((p - (float)top) + e) : 0;
    }
#pragma unroll
    for (int h = 0; h < oz::DCOL / 8; h++)
#pragma unroll
      for (int s = NS - 1; s >= 0; s--) {
        uint4 w;
        w.x = oz::digit_pair32(f[8 * h], f[8 * h + 1], s);
        w.y = oz::digit_pair32(f[8 * h + 2], f[8 * h + 3], s);
        w.z = oz::digit_pair32(f[8 * h + 4], f[8 * h + 5], s);
        w.w = oz::digit_pair32(f[8 * h + 6], f[8 * h + 7], s);
        *reinterpret_cast<uint4*>(o + s * slice + 8 * h) = w;
        if (tail) *reinterpret_cast<uint4*>(o + s * slice + 16 + 8 * h) = make_uint4(0, 0, 0, 0);
      }
  }
};
// C = sum Sigma W as double-float pairs, out[row][col].
struct OzEpiC {
  static constexpr bool kWarp = false, kDigits = false, kPair = true, kLong = true;
  const int* eP;
  using Scale = float;
  __device__ __forceinline__ float scale(const oz::Job& jb) const {
    const int ep = eP[jb.o_e];
    if (ep > oz::EX_NAN / 2) return __int_as_float(0x7FC00000);
    return ep < -100 ? 0.f : __int_as_float((1 + ep - 14 + 127) << 23);
  }
  __device__ __forceinline__ void tile(const oz::Job& jb, float sc, int r, int c0, const float (&vh)[oz::DCOL],
                                       const float (&vl)[oz::DCOL]) const {
    dfl* o = static_cast<dfl*>(jb.out) + (size_t)(jb.m0 + r) * jb.ld_out + jb.n0 + c0;
#pragma unroll
    for (int u = 0; u < oz::DCOL; u++)
      if (c0 + u < jb.n_valid) o[u] = df_norm(vh[u] * sc, vl[u] * sc);
  }
};
// T_ii from FP32 pairs (mixed form).
struct OzEpiTPair {
  static constexpr bool kWarp = false, kDigits = false, kPair = true, kLong = false;
  const double* e_vir;
  __device__ __forceinline__ void pairs(const oz::Job& jb, int r, int c0, const float (&h)[oz::DCOL],
                                        const float (&l)[oz::DCOL]) const {
    double v[oz::DCOL];
#pragma unroll
    for (int u = 0; u < oz::DCOL; u++) v[u] = (double)h[u] + (double)l[u];
    OzEpiT{e_vir}(jb, r, c0, v);
  }
};

// Digits of the output instead of its values: row m0 + r, k = n0 + c of the matrix at store row o_row, under the exponent code exW[o_e] (a bound of the whole matrix); columns past n_valid up to the
// next multiple of 16 are written as zeros (up to 32 by the lanes of the last column group).
template <int NS>
struct OzEpiDigits {
  static constexpr bool kWarp = false, kDigits = true, kPair = false, kLong = false;
  static constexpr int T = 7 + 8 * (NS - 1);
  uint16_t* D;
  int ld;
  size_t slice;
  const int* exW;
  __device__ __forceinline__ int exponent(const oz::Job& jb) const { return exW[jb.o_e]; }
  __device__ __forceinline__ void digits(const oz::Job& jb, int r, int c0, long long (&f)[oz::DCOL]) const {
    uint16_t* o = D + ((size_t)jb.o_row + jb.m0 + r) * ld + jb.n0 + c0;
    // the last column group also clears the group after it when that completes a 32-wide k-block
    const bool tail = c0 + oz::DCOL >= jb.n_valid && ((jb.n0 + c0) & 16) == 0;
#pragma unroll
    for (int u = 0; u < oz::DCOL; u++)
      if (c0 + u >= jb.n_valid) f[u] = 0;
#pragma unroll
    for (int h = 0; h < oz::DCOL / 8; h++)
#pragma unroll
      for (int s = NS - 1; s >= 0; s--) {
        uint4 w;
        w.x = oz::digit_pair(f[8 * h], f[8 * h + 1], s);
        w.y = oz::digit_pair(f[8 * h + 2], f[8 * h + 3], s);
        w.z = oz::digit_pair(f[8 * h + 4], f[8 * h + 5], s);
        w.w = oz::digit_pair(f[8 * h + 6], f[8 * h + 7], s);
        *reinterpret_cast<uint4*>(o + s * slice + 8 * h) = w;
        if (tail) *reinterpret_cast<uint4*>(o + s * slice + 16 + 8 * h) = make_uint4(0, 0, 0, 0);
      }
  }
};

// <2 Y - Y^T, D> of the tile's part of D (never stored): Y = the r x r matrix at job.out (r = ld_out), one
// partial sum per drain warp at parts + 16 job.o_row.
struct OzEpiDot {
  static constexpr bool kWarp = true, kDigits = false, kPair = false, kLong = false;
  double* parts;
  __device__ __forceinline__ void warp(const oz::Job& jb, int r, int c0, const double (&v)[oz::DCOL]) const {
    const double* Y = static_cast<const double*>(jb.out);
    double s = 0.0;
    if (r < jb.m_valid) {
      const int a = jb.m0 + r;
#pragma unroll
      for (int u = 0; u < oz::DCOL; u++) {
        const int b = jb.n0 + c0 + u;
        if (c0 + u < jb.n_valid) s += (2.0 * Y[(size_t)a * jb.ld_out + b] - Y[(size_t)b * jb.ld_out + a]) * v[u];
      }
    }
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) parts[(size_t)oz::NDRAIN * jb.o_row + (threadIdx.x >> 5) - 2] = s;
  }
};

// Sum of the squares of the tile's part of D (never stored), one partial sum per drain warp at parts + 16 job.o_row.
struct OzEpiSquares {
  static constexpr bool kWarp = true, kDigits = false, kPair = false, kLong = false;
  double* parts;
  __device__ __forceinline__ void warp(const oz::Job& jb, int r, int c0, const double (&v)[oz::DCOL]) const {
    double s = 0.0;
    if (r < jb.m_valid) {
#pragma unroll
      for (int u = 0; u < oz::DCOL; u++)
        if (c0 + u < jb.n_valid) s = fma(v[u], v[u], s);
    }
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) parts[(size_t)oz::NDRAIN * jb.o_row + (threadIdx.x >> 5) - 2] = s;
  }
};

namespace {
// 3-D BF16 map over k x rows x slices, 64-byte swizzle, box 32 x box_rows x ns.  K < ld: k past K reads as 0.
bool make_digit_map(CUtensorMap* m, const OzOperand& A, int ns, int box_rows) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)A.K, (cuuint64_t)A.rows, (cuuint64_t)ns};
  cuuint64_t strides[2] = {(cuuint64_t)A.ld * 2, (cuuint64_t)A.rows * A.ld * 2};
  cuuint32_t box[3] = {(cuuint32_t)oz::BK, (cuuint32_t)box_rows, (cuuint32_t)ns};
  cuuint32_t es[3] = {1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<uint16_t*>(A.D), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int NS, class Epi>
int run(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs, const int* skip,
        int* err, Epi epi, cudaStream_t st) {
  if (!n_jobs) return 0;
  constexpr int SMEM = oz::Cfg<NS>::SMEM;
  if (cudaFuncSetAttribute(oz::k_oz<NS, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM) != cudaSuccess) return -1;
  oz::OzMaps tm;
  for (int u = 0; u < 2; u++)
    if (!make_digit_map(&tm.a[u], A, NS, oz::BM >> (1 - u)) || !make_digit_map(&tm.b[u], B, NS, oz::tile_cols(NS) >> (1 - u))) return -1;
  oz::k_oz<NS, Epi><<<tc::persistent_grid(n_jobs), oz::NTHREADS, SMEM, st>>>(tm, A.ex, B.ex, jobs, n_jobs, segs, skip,
                                                                             err, epi);
  note_launch(1);
  return 0;
}
}  // namespace

int launch_oz_gemm(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                   const int* skip, int* err, cudaStream_t st) {
  return run<oz::NSL>(A, B, jobs, n_jobs, segs, skip, err, OzEpiRow{}, st);
}
int launch_oz_digits(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                     const int* skip, uint16_t* D, int ld, long long rows, const int* exW, int* err, cudaStream_t st) {
  return run<oz::NSL>(A, B, jobs, n_jobs, segs, skip, err, OzEpiDigits<oz::NSL>{D, ld, (size_t)rows * ld, exW}, st);
}
int launch_mx_w(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                const int* skip, uint16_t* D, int ld, long long rows, const int* eY, const int* eP, int* err,
                cudaStream_t st) {
  return run<oz::MXSOLVE>(A, B, jobs, n_jobs, segs, skip, err, OzEpiW{D, ld, (size_t)rows * ld, eY, eP}, st);
}
int launch_mx_c(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                const int* skip, const int* eP, int* err, cudaStream_t st) {
  return run<oz::MXSOLVE>(A, B, jobs, n_jobs, segs, skip, err, OzEpiC{eP}, st);
}
int launch_mx_g(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                long long lo_shift, int* err, cudaStream_t st) {
  return run<oz::MXSL>(A, B, jobs, n_jobs, segs, nullptr, err, OzEpiG{lo_shift}, st);
}
int launch_mx_gemm(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                   bool fp64_out, int* err, cudaStream_t st) {
  return fp64_out ? run<oz::MXSL>(A, B, jobs, n_jobs, segs, nullptr, err, OzEpiPair<double>{}, st)
                  : run<oz::MXSL>(A, B, jobs, n_jobs, segs, nullptr, err, OzEpiPair<float>{}, st);
}
int launch_oz_dots(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                   double* parts, int* err, cudaStream_t st) {
  return run<8>(A, B, jobs, n_jobs, segs, nullptr, err, OzEpiDot{parts}, st);
}
int launch_oz_squares(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                      double* parts, int* err, cudaStream_t st) {
  return run<oz::NSL>(A, B, jobs, n_jobs, segs, nullptr, err, OzEpiSquares{parts}, st);
}
int launch_oz_tii(const OzOperand& A, const oz::Job* jobs, int n_jobs, const oz::Seg* segs, const double* e_vir, int ns,
                  int* err, cudaStream_t st) {
  return ns == oz::NSL ? run<oz::NSL>(A, A, jobs, n_jobs, segs, nullptr, err, OzEpiT{e_vir}, st)
                       : run<oz::MXSL>(A, A, jobs, n_jobs, segs, nullptr, err, OzEpiTPair{e_vir}, st);
}

}  // namespace osv

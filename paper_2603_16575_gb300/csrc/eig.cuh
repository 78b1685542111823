// CTA-wide FP64 symmetric eigen-solvers used by the OSV build (Eq. osv_gen)
// and by the pair preconditioner (Eq. prec_eig).
//
//  * cta_tridiag     Householder reduction A = Z T Z^T to tridiagonal form
//                    (reflectors H_k = I - tau_k v_k v_k^T, v_k[0] = 1, stored
//                    below the sub-diagonal of A).
//  * cta_form_z      Z = H_0 H_1 ... H_{n-3} by backward accumulation.
//  * cta_tridiag_qr  implicit symmetric QR steps with the Wilkinson shift
//                    (Golub & Van Loan, Matrix Computations, Alg. 8.3.2/8.3.3),
//                    rotations accumulated into the columns of Z.
//  * sturm_count / multisection / inverse iteration + back-transformation for the
//    eigenpairs above a threshold, used when only a few OSVs out of a large
//    virtual space are kept.
// All routines are called by every thread of a CTA of NT threads.
#pragma once
#include "common.cuh"

namespace osv {

// FP32 seeds of FP64 reciprocals and roots by integer operations (a conversion holds the FP64 pipe as an FMA does).
__device__ __forceinline__ float mant_f(int hi, int lo) {          // the float below a double in [1, 4)
  return __int_as_float((((hi >> 20) - 1023 + 127) << 23) | ((hi & 0xfffff) << 3) | (int)((unsigned)lo >> 29));
}
__device__ __forceinline__ double widen(float f, int de) {         // f 2^de, f normal and positive, by integer operations
  const int b = __float_as_int(f);
  return __hiloint2double(((b >> 23) - 127 + 1023 + de) << 20 | (b & 0x7fffff) >> 3, b << 29);
}
// s^(-1/2) for s > 0: the FP32 reciprocal root of the mantissa refined by one step of third order (Halley; error
// ~2^-60 before rounding), six FP64 operations; near the ends of the range by the library's function.
__device__ __forceinline__ double rsqrt_halley(double s) {
  const int hi = __double2hiint(s), lo = __double2loint(s), ex = (hi >> 20) & 2047;
  if (ex < 64 || ex > 1983) return rsqrt(s);
  const int q = (ex - 1023) >> 1;                                  // s = m 4^q, m in [1, 4)
  const double m = __hiloint2double(hi - (q << 21), lo);
  const double r0 = widen(rsqrtf(mant_f(hi - (q << 21), lo)), 0);
  const double e = fma(-m * r0, r0, 1.0);
  const double r = fma(r0 * e, fma(e, 0.375, 0.5), r0);
  return __hiloint2double(__double2hiint(r) - (q << 20), __double2loint(r));
}

// Householder tridiagonalisation of the symmetric n x n matrix A (row-major,
// lda; global or shared memory), in place.  Outputs d[n], e[n-1] (any memory)
// and tau[n]; v and p are shared scratch of n elements each, red >= 33.
// T = double or float.
template <int NTH = NT, class T = double>
__device__ inline void cta_tridiag(T* A, int n, int lda, T* d, T* e, T* tau, T* v, T* p, T* red) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = NTH / 32;
  __shared__ T s_tau;
  for (int k = 0; k + 2 < n; k++) {
    const int L = n - k - 1;          // trailing block rows/cols k+1 .. n-1
    T* Ak = A + (size_t)(k + 1) * lda + (k + 1);   // trailing block origin
    T part = T(0.0);
    for (int t = tid; t < L; t += NTH) {
      const T x = A[(size_t)(k + 1 + t) * lda + k];
      v[t] = x;
      if (t > 0) part += x * x;
    }
    const T sigma = cta_sum(part, red);
    if (tid == 0) {
      const T alpha = v[0];
      T tu = T(0.0), beta = alpha;
      if (sigma > T(0.0)) {
        const T mu = sqrt(alpha * alpha + sigma);
        beta = alpha <= T(0.0) ? mu : -mu;
        tu = (beta - alpha) / beta;
        const T v0 = alpha - beta;
        red[0] = T(1.0) / v0;   // scale for v[1..]
      }
      s_tau = tu;
      d[k] = A[(size_t)k * lda + k];
      e[k] = beta;
      tau[k] = tu;
    }
    __syncthreads();
    const T tk = s_tau;
    if (tk != T(0.0)) {
      const T sc = red[0];
      for (int t = tid; t < L; t += NTH) v[t] = (t == 0) ? T(1.0) : v[t] * sc;
      __syncthreads();
      // p = tau * A' v  (warp per row, lanes over columns)
      for (int r = warp; r < L; r += nwarp) {
        const T* row = Ak + (size_t)r * lda;
        T s0 = T(0.0), s1 = T(0.0), s2 = T(0.0), s3 = T(0.0);
        int c = lane;
        for (; c + 96 < L; c += 128) {       // four independent loads in flight per lane
          const T a0 = row[c], a1 = row[c + 32], a2 = row[c + 64], a3 = row[c + 96];
          s0 += a0 * v[c];
          s1 += a1 * v[c + 32];
          s2 += a2 * v[c + 64];
          s3 += a3 * v[c + 96];
        }
        for (; c < L; c += 32) s0 += row[c] * v[c];
        const T s = warp_sum((s0 + s1) + (s2 + s3));
        if (lane == 0) p[r] = tk * s;
      }
      __syncthreads();
      T pv = T(0.0);
      for (int t = tid; t < L; t += NTH) pv += p[t] * v[t];
      const T Kc = T(0.5) * tk * cta_sum(pv, red);
      for (int t = tid; t < L; t += NTH) p[t] -= Kc * v[t];   // p becomes w
      __syncthreads();
      // A' -= v w^T + w v^T
      for (int r = warp; r < L; r += nwarp) {
        T* row = Ak + (size_t)r * lda;
        const T vr = v[r], wr = p[r];
        int c = lane;
        for (; c + 96 < L; c += 128) {
          const T a0 = row[c], a1 = row[c + 32], a2 = row[c + 64], a3 = row[c + 96];
          row[c] = a0 - (vr * p[c] + wr * v[c]);
          row[c + 32] = a1 - (vr * p[c + 32] + wr * v[c + 32]);
          row[c + 64] = a2 - (vr * p[c + 64] + wr * v[c + 64]);
          row[c + 96] = a3 - (vr * p[c + 96] + wr * v[c + 96]);
        }
        for (; c < L; c += 32) row[c] -= vr * p[c] + wr * v[c];
      }
      // keep the reflector below the sub-diagonal of column k
      for (int t = tid + 1; t < L; t += NTH) A[(size_t)(k + 1 + t) * lda + k] = v[t];
    }
    __syncthreads();
  }
  if (tid == 0) {
    if (n >= 2) {
      d[n - 2] = A[(size_t)(n - 2) * lda + (n - 2)];
      e[n - 2] = A[(size_t)(n - 1) * lda + (n - 2)];
      if (n >= 3) tau[n - 2] = T(0.0);
    }
    d[n - 1] = A[(size_t)(n - 1) * lda + (n - 1)];
    tau[n - 1] = T(0.0);
  }
  __syncthreads();
}

// Z (n x n, row-major, ldz) = H_0 H_1 ... H_{n-3} from the reflectors left in A.
// y, vs: shared scratch of n doubles each.
template <int NTH = NT>
__device__ inline void cta_form_z(const double* A, int n, int lda, const double* tau, double* Z, int ldz,
                                  double* y, double* vs) {
  const int tid = threadIdx.x;
  for (int t = tid; t < n * n; t += NTH) Z[(size_t)(t / n) * ldz + (t % n)] = (t / n == t % n) ? 1.0 : 0.0;
  __syncthreads();
  for (int k = n - 3; k >= 0; k--) {
    const double tk = tau[k];
    if (tk == 0.0) continue;
    const int L = n - k - 1;
    for (int r = tid; r < L; r += NTH) vs[r] = (r == 0) ? 1.0 : A[(size_t)(k + 1 + r) * lda + k];
    __syncthreads();
    // y_c = tau * sum_r v_r Z[k+1+r][k+1+c]
    for (int c = tid; c < L; c += NTH) {
      double s = 0.0;
      for (int r = 0; r < L; r++) s += vs[r] * Z[(size_t)(k + 1 + r) * ldz + (k + 1 + c)];
      y[c] = tk * s;
    }
    __syncthreads();
    for (int t = tid; t < L * L; t += NTH) {
      const int r = t / L, c = t % L;
      Z[(size_t)(k + 1 + r) * ldz + (k + 1 + c)] -= vs[r] * y[c];
    }
    __syncthreads();
  }
}

// Implicit symmetric QR on the tridiagonal (d[n], e[n-1]) with rotations
// accumulated into the columns of Z (n x n, row-major, ldz).  d, e must be in
// shared or global memory visible to thread 0; cs is shared scratch of 2n
// elements.  Returns 0 on convergence (d holds the eigenvalues, columns of Z the
// eigenvectors), 1 otherwise.  Every thread returns the same value.
// ZCM: Z stored column-major (Z[r][c] at Z[c * ldz + r]), so that the threads,
// one per row, rotate it with coalesced accesses.  T = double or float.
template <int NTH = NT, bool ZCM = false, class T = double>
__device__ inline int cta_tridiag_qr(T* d, T* e, int n, T* Z, int ldz, T* cs) {
  __shared__ int s_l, s_h, s_done;
  const int tid = threadIdx.x;
  const T eps = sizeof(T) == 8 ? T(2.220446049250313e-16) : T(1.1920929e-07);
  int sweeps = 0;
  const int max_sweeps = 40 * n + 100;
  while (true) {
    if (tid == 0) {
      int h = n - 1, l = 0, done = 0;
      // deflate negligible couplings from the bottom
      while (h > 0) {
        if (fabs(e[h - 1]) <= eps * (fabs(d[h - 1]) + fabs(d[h]))) { e[h - 1] = T(0.0); h--; }
        else break;
      }
      if (h == 0) done = 1;
      else {
        l = h - 1;
        while (l > 0) {
          if (fabs(e[l - 1]) <= eps * (fabs(d[l - 1]) + fabs(d[l]))) { e[l - 1] = T(0.0); break; }
          l--;
        }
        // Wilkinson shift from the trailing 2x2 of the unreduced block [l, h]
        const T delta = T(0.5) * (d[h - 1] - d[h]);
        const T eh = e[h - 1];
        const T den = delta + copysign(hypot(delta, eh), delta);
        const T mu = d[h] - (den != T(0.0) ? eh * eh / den : T(0.0));
        T x = d[l] - mu, z = e[l];
        for (int k = l; k < h; k++) {
          const T r = hypot(x, z);
          T c = T(1.0), s = T(0.0);
          if (r != T(0.0)) { c = x / r; s = z / r; }
          if (k > l) e[k - 1] = r;
          const T a = d[k], b = e[k], cc = d[k + 1];
          d[k] = c * c * a + T(2.0) * c * s * b + s * s * cc;
          d[k + 1] = s * s * a - T(2.0) * c * s * b + c * c * cc;
          e[k] = c * s * (cc - a) + (c * c - s * s) * b;
          if (k + 1 < h) {
            x = e[k];
            z = s * e[k + 1];
            e[k + 1] = c * e[k + 1];
          }
          cs[2 * k] = c;
          cs[2 * k + 1] = s;
        }
      }
      s_l = l; s_h = h; s_done = done;
    }
    __syncthreads();
    if (s_done) return 0;
    if (++sweeps > max_sweeps) return 1;
    const int l = s_l, h = s_h;
    // Z <- Z R_l^T R_{l+1}^T ... : column pair (k, k+1) rotated for k = l..h-1
    for (int row = tid; row < n; row += NTH) {
      T* zr = ZCM ? Z + row : Z + (size_t)row * ldz;
      const size_t zs = ZCM ? (size_t)ldz : 1;   // stride between the columns of one row
      T carry = zr[l * zs];
      for (int k = l; k < h; k++) {
        const T c = cs[2 * k], s = cs[2 * k + 1];
        const T y = zr[(k + 1) * zs];
        zr[k * zs] = c * carry + s * y;
        carry = -s * carry + c * y;
      }
      zr[h * zs] = carry;
    }
    __syncthreads();
  }
}

// Full symmetric eigen-decomposition of A (n x n, row-major lda, destroyed).
// On return w[0..n) holds the eigenvalues and column t of Z the eigenvector
// of w[t] (unordered).  d/e/tau: n doubles each (any memory visible to the
// CTA); sm: shared scratch of >= 4n + 33 doubles.  Returns 0 on success.
template <int NTH = NT>
__device__ inline int cta_syev(double* A, int n, int lda, double* w, double* Z, int ldz, double* e,
                               double* tau, double* sm) {
  double* v = sm;
  double* p = sm + n;
  double* cs = sm + 2 * n;      // 2n
  double* red = sm + 4 * n;     // 33
  if (n == 1) {
    if (threadIdx.x == 0) { w[0] = A[0]; Z[0] = 1.0; }
    __syncthreads();
    return 0;
  }
  cta_tridiag<NTH>(A, n, lda, w, e, tau, v, p, red);
  cta_form_z<NTH>(A, n, lda, tau, Z, ldz, v, p);
  // the bulge chase is sequential: run it on shared-memory copies of d and e
  for (int t = threadIdx.x; t < n; t += NTH) {
    v[t] = w[t];
    p[t] = (t + 1 < n) ? e[t] : 0.0;
  }
  __syncthreads();
  const int rc = cta_tridiag_qr<NTH>(v, p, n, Z, ldz, cs);
  for (int t = threadIdx.x; t < n; t += NTH) w[t] = v[t];
  __syncthreads();
  return rc;
}

// Z = H_0 H_1 ... H_{n-3} from the reflectors left in A, stored column-major
// (Z[r][c] at Z[c * ldz + r]); a warp per column forms the dot products along
// contiguous memory.  y, vs: shared scratch of n elements each.
// T = double or float.  ROWV: reflector k in row k to the right of the diagonal
// (k_eig_tri) instead of below the sub-diagonal of column k (cta_tridiag).
template <int NTH = NT, class T, bool ROWV = false>
__device__ inline void cta_form_z_cm(const T* A, int n, int lda, const T* tau, T* Z, int ldz, T* y, T* vs) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = NTH / 32;
  for (int t = tid; t < n * n; t += NTH) Z[(size_t)(t / n) * ldz + (t % n)] = (t / n == t % n) ? T(1.0) : T(0.0);
  __syncthreads();
  for (int k = n - 3; k >= 0; k--) {
    const T tk = tau[k];
    if (tk == T(0.0)) continue;
    const int L = n - k - 1;
    for (int r = tid; r < L; r += NTH)
      vs[r] = (r == 0) ? T(1.0) : (ROWV ? A[(size_t)k * lda + k + 1 + r] : A[(size_t)(k + 1 + r) * lda + k]);
    __syncthreads();
    // y_c = tau * sum_r v_r Z[k+1+r][k+1+c]: column k+1+c is contiguous
    for (int c = warp; c < L; c += NW) {
      const T* zc = Z + (size_t)(k + 1 + c) * ldz + (k + 1);
      T s = T(0.0);
      for (int r = lane; r < L; r += 32) s = fma(vs[r], zc[r], s);
      s = warp_sum(s);
      if (lane == 0) y[c] = tk * s;
    }
    __syncthreads();
    for (int t = tid; t < L * L; t += NTH) {
      const int c = t / L, r = t % L;
      Z[(size_t)(k + 1 + c) * ldz + (k + 1 + r)] -= vs[r] * y[c];
    }
    __syncthreads();
  }
}

// Full symmetric eigen-decomposition as cta_syev with Z column-major: on
// return w[0..n) holds the eigenvalues and Z[t * ldz + a] is component a of
// the eigenvector of w[t] (unordered).  A (row-major, lda) is destroyed; e,
// tau: n elements each (any memory visible to the CTA); sm: shared scratch of
// >= 4n + 33 elements.  Returns 0 on success.  T = double or float.
template <int NTH = NT, class T>
__device__ inline int cta_syev_cm(T* A, int n, int lda, T* w, T* Z, int ldz, T* e, T* tau, T* sm) {
  T* v = sm;
  T* p = sm + n;
  T* cs = sm + 2 * n;      // 2n
  T* red = sm + 4 * n;     // 33
  if (n == 1) {
    if (threadIdx.x == 0) { w[0] = A[0]; Z[0] = T(1.0); }
    __syncthreads();
    return 0;
  }
  cta_tridiag<NTH>(A, n, lda, w, e, tau, v, p, red);
  cta_form_z_cm<NTH>(A, n, lda, tau, Z, ldz, v, p);
  for (int t = threadIdx.x; t < n; t += NTH) {   // the bulge chase runs on shared copies of d and e
    v[t] = w[t];
    p[t] = (t + 1 < n) ? e[t] : T(0.0);
  }
  __syncthreads();
  const int rc = cta_tridiag_qr<NTH, true>(v, p, n, Z, ldz, cs);
  for (int t = threadIdx.x; t < n; t += NTH) w[t] = v[t];
  __syncthreads();
  return rc;
}

// ---------------------------------------------------------------- batched QR
// The bulge chase of the implicit QR (as cta_tridiag_qr) is sequential; run by
// one thread of a CTA it leaves the rest of the CTA idle and, in FP64, uses a
// thirty-second of the FP64 pipe for every instruction.  These two routines
// split cta_tridiag_qr into (a) the chase of one tridiagonal per THREAD, many
// problems per warp, recording the sweeps (l, h) and their rotations, and (b)
// the application of the recorded rotations to the rows of Z by a CTA.  The
// sweeps are those of cta_tridiag_qr; the rotations are formed with fewer
// FP64 operations, since each holds the pipe 64 cycles however few lanes work:
// ~20 a rotation in place of ~28 (chase_rotation by rsqrt_halley, a shared
// term in the update, exponents in the tests for zero).

// (a) One thread: chase (d[n], e[n-1]) to diagonal form, appending each sweep
// to swp (l, h pairs, capacity cap_s sweeps) and its rotations (c, s pairs,
// capacity cap_r) to rot.  Returns 0 on convergence (*n_sw sweeps recorded, d
// holds the eigenvalues), 1 if the sweep limit was reached, 2 if a record
// would overflow.  With partial, the overflow return also sets *n_sw to the
// sweeps recorded so far (d, e are then those after them, so a later call
// continues the chase).
// Givens rotation (c, s) with c x + s z = r >= 0, -s x + c z = 0.  FP64: one
// reciprocal square root; FP32: a correctly rounded square root and one
// division (unbiased rounding, so the accumulated rotations stay orthogonal
// to the FP32 rounding level).  hypot and two divisions where x^2 + z^2 could
// leave the normal range.
__device__ __forceinline__ void chase_rotation(double x, double z, double& c, double& s, double& r) {
  const double q = fma(z, z, x * x);
  const int ex = (__double2hiint(q) >> 20) & 2047;
  if (ex > 93 && ex < 1953) {     // 1e-280 .. 1e280
    const double inv = rsqrt_halley(q);
    c = x * inv;
    s = z * inv;
    r = q * inv;
  } else {
    r = hypot(x, z);
    c = 1.0;
    s = 0.0;
    if (r != 0.0) { c = x / r; s = z / r; }
  }
}
__device__ __forceinline__ void chase_rotation(float x, float z, float& c, float& s, float& r) {
  const float q = x * x + z * z;
  if (q > 1e-36f && q < 1e36f) {
    r = sqrtf(q);
    const float inv = 1.f / r;
    c = x * inv;
    s = z * inv;
  } else {
    r = hypotf(x, z);
    c = 1.f;
    s = 0.f;
    if (r != 0.f) { c = x / r; s = z / r; }
  }
}

// |e| <= eps (|d0| + |d1|); in FP64 the exponents decide for the entries far above it (eps = 2^-52, so
// |e| >= 2^-49 max |d| is not; no FP64 operation); zeros take the comparison.
template <class T>
__device__ __forceinline__ bool off_negligible(T e, T d0, T d1, T eps) {
  if constexpr (sizeof(T) == 8) {
    const int xe = (__double2hiint(e) >> 20) & 2047;
    const int xd = max((__double2hiint(d0) >> 20) & 2047, (__double2hiint(d1) >> 20) & 2047);
    if (xe > 0 && xe > xd - 50) return false;
  }
  return fabs(e) <= eps * (fabs(d0) + fabs(d1));
}

// S: stride of d and e (one tridiagonal per lane, interleaved in shared memory).
template <int S = 1, class T>
__device__ inline int tridiag_qr_record(T* __restrict__ d, T* __restrict__ e, int n, int* __restrict__ swp, int cap_s,
                                        T* __restrict__ rot, int cap_r, int* n_sw, bool partial = false) {
  const T eps = sizeof(T) == 8 ? T(2.220446049250313e-16) : T(1.1920929e-07);
  const int max_sweeps = 40 * n + 100;
  int ns = 0, nr = 0;
  *n_sw = 0;
  for (int sweeps = 0;; sweeps++) {
    int h = n - 1;
    while (h > 0) {
      if (off_negligible(e[(h - 1) * S], d[(h - 1) * S], d[(h) * S], eps)) { e[(h - 1) * S] = T(0.0); h--; }
      else break;
    }
    if (h == 0) { *n_sw = ns; return 0; }
    if (sweeps >= max_sweeps) return 1;
    int l = h - 1;
    while (l > 0) {
      if (off_negligible(e[(l - 1) * S], d[(l - 1) * S], d[(l) * S], eps)) { e[(l - 1) * S] = T(0.0); break; }
      l--;
    }
    if (ns >= cap_s || nr + (h - l) > cap_r) {
      if (partial) *n_sw = ns;
      return 2;
    }
    swp[2 * ns] = l;
    swp[2 * ns + 1] = h;
    ns++;
    T* cs = rot + 2 * (size_t)nr;
    nr += h - l;
    const T delta = T(0.5) * (d[(h - 1) * S] - d[(h) * S]);
    const T eh = e[(h - 1) * S];
    const T den = delta + copysign(hypot(delta, eh), delta);
    const T mu = d[(h) * S] - (den != T(0.0) ? eh * eh / den : T(0.0));
    // d[(k) * S] and e[(k) * S] as updated by the previous rotation stay in registers
    T dk = d[(l) * S], ek = e[(l) * S];
    T x = dk - mu, z = ek;
    for (int k = l; k < h; k++) {
      const T cc = d[(k + 1) * S];
      const T en = (k + 1 < h) ? e[(k + 1) * S] : T(0.0);
      T c, s, r;
      chase_rotation(x, z, c, s, r);
      if (k > l) e[(k - 1) * S] = r;
      // c^2 a + 2 c s b + s^2 cc = a + s h, s^2 a - 2 c s b + c^2 cc = cc - s h, c s (cc - a) + (c^2 - s^2) b = c h - b
      // with h = s (cc - a) + 2 c b: eight operations of a chain that one thread walks
      const T a = dk, b = ek, h2 = fma(s, cc - a, (c + c) * b), p = s * h2;
      d[(k) * S] = a + p;
      dk = cc - p;
      const T ekn = fma(c, h2, -b);
      e[(k) * S] = ekn;
      if (k + 1 < h) {
        x = ekn;
        z = s * en;
        ek = c * en;
      }
      cs[2 * (k - l)] = c;
      cs[2 * (k - l) + 1] = s;
    }
    d[(h) * S] = dk;
  }
}

// (b) The CTA: apply the n_sw recorded sweeps to Z (n x n, column-major, ldz;
// a thread per row, coalesced).
template <int NTH = NT, class T>
__device__ inline void apply_qr_record_cm(T* Z, int ldz, int n, const int* swp, int n_sw, const T* rot) {
  for (int row = threadIdx.x; row < n; row += NTH) {
    T* zr = Z + row;
    const T* cs = rot;
    for (int q = 0; q < n_sw; q++) {
      const int l = swp[2 * q], h = swp[2 * q + 1];
      T carry = zr[(size_t)l * ldz];
      for (int k = l; k < h; k++, cs += 2) {
        const T c = cs[0], s = cs[1];
        const T y = zr[(size_t)(k + 1) * ldz];
        zr[(size_t)k * ldz] = c * carry + s * y;
        carry = -s * carry + c * y;
      }
      zr[(size_t)h * ldz] = carry;
    }
  }
  __syncthreads();
}

// ---------------------------------------------------------------- top-k
// Number of eigenvalues of the tridiagonal (d, e) strictly below x: sign changes of the leading principal minors
// of T - x I by their three-term recurrence, one FMA of chain a row (the LDL^T pivots, the ratios of the minors,
// take an FP64 division a row, ~10 operations; an FP64 operation of a warp holds its sub-partition's pipe
// for 64 cycles, so their number is the time).  The rounding is that of a relative change of d - x and e by a few
// eps, as with the pivots.  ||T|| <= 1 (the caller scales by a power of two), so four rows grow a minor by
// < 2^7; the two live ones are rescaled every four rows.  e2[i] = e[i]^2, at least 1e-60: no two
// successive minors vanish, and the sign of a single zero does not change the count.
__device__ __forceinline__ int sturm_count_minors(const double* d, const double* e2, int n, double x) {
  double p0 = 0.0, p1 = 1.0;
  int cnt = 0;
  for (int i0 = 0; i0 < n; i0 += 4) {
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const int i = i0 + u;
      if (i < n) {
        const double ep = e2[i > 0 ? i - 1 : 0] * p0;
        const double p = fma(d[i] - x, p1, -ep);
        cnt += (__double2hiint(p) ^ __double2hiint(p1)) < 0;
        p0 = p1;
        p1 = p;
      }
    }
    const int ex = max((__double2hiint(p0) >> 20) & 2047, (__double2hiint(p1) >> 20) & 2047);
    const double sc = __hiloint2double(min(2046, max(1, 2046 - ex)) << 20, 0);   // 2^(1023 - ex)
    p0 *= sc;
    p1 *= sc;
  }
  return cnt;
}
// Eigenvalues with ascending indices n-1-t, t < k, of (d, e) by multisection
// on the Sturm count, called by one warp that handles t = t0, t0 + tstride, ...:
// g = lane / L lanes per eigenvalue split its interval at L points per step
// (log2(L+1) bits per Sturm sequence instead of one), until the interval is
// below 2 eps |lambda| or atol (the eigenvalues of the tridiagonal are only
// determined to ~eps ||T|| by its rounding).  w[t] receives the eigenvalue times wscale.
__device__ inline void multisect_eigs(const double* d, const double* e2, int n, int k, int t0, int tstride,
                                      double lo0, double hi0, double atol, double wscale, double* w) {
  const int lane = threadIdx.x & 31;
  const int ng = (k - t0 + tstride - 1) / tstride;   // eigenvalues of this warp
  if (ng <= 0) return;
  const int L = max(1, 32 / ng);
  const int gmax = 32 / L;                                  // groups per pass
  const double eps = 2.220446049250313e-16;
  for (int gb = 0; gb < ng; gb += gmax) {
    const int g = gb + lane / L, q = lane % L;
    const int t = t0 + g * tstride;
    const bool mine = (lane / L < gmax) && (g < ng) && (t < k);
    const int j = n - 1 - t;
    double lo = lo0, hi = hi0;
    bool done = !mine;
    for (int it = 0; it < 200; it++) {
      if (!__any_sync(0xffffffffu, !done)) break;
      const double x = lo + (hi - lo) * (double)(q + 1) / (double)(L + 1);
      bool above = false;   // more than j eigenvalues below x: eigenvalue j lies below x
      if (!done) above = sturm_count_minors(d, e2, n, x) > j;
      const unsigned bal = __ballot_sync(0xffffffffu, above);
      if (!done) {
        const unsigned bits = (bal >> ((lane / L) * L)) & ((L == 32) ? 0xffffffffu : ((1u << L) - 1u));
        const int qs = bits ? (__ffs(bits) - 1) : L;        // first split point above eigenvalue j
        const double nlo = (qs == 0) ? lo : lo + (hi - lo) * (double)qs / (double)(L + 1);
        const double nhi = (qs == L) ? hi : lo + (hi - lo) * (double)(qs + 1) / (double)(L + 1);
        if (!(nlo > lo || nhi < hi)) done = true;           // no progress at this precision
        lo = nlo;
        hi = nhi;
        if (hi - lo <= fmax(2.0 * eps * fmax(fabs(lo), fabs(hi)), atol)) done = true;
      }
    }
    if (mine && q == 0) w[t] = 0.5 * (lo + hi) * wscale;
  }
  __syncwarp();
}

// a / b in double-float: an FP32 quotient corrected once with the exact
// remainder (~2^-46 relative).
__device__ __forceinline__ dfl df_div(dfl a, dfl b) {
  const float q1 = __fdividef(a.h, b.h);
  const dfl r = df_add(a, df_neg(df_mul(dfl{q1, 0.f}, b)));
  const float q2 = __fdividef(r.h, b.h);
  return df_fast2(q1, q2);
}
// Sturm count by the LDL^T pivots in double-float: d and e^2 as (hi, lo) pairs, x converted once;
// pivmin in FP32 range.
__device__ inline int sturm_count_df(const dfl* d, const dfl* e2, int n, double x, float pivmin) {
  const dfl nx = df_neg(df_from(x));
  int cnt = 0;
  dfl q = df_add(d[0], nx);
  if (fabsf(q.h) < pivmin) q = dfl{-pivmin, 0.f};
  cnt += q.h < 0.f;
  for (int i = 1; i < n; i++) {
    q = df_add(df_add(d[i], nx), df_neg(df_div(e2[i - 1], q)));
    if (fabsf(q.h) < pivmin) q = dfl{-pivmin, 0.f};
    cnt += q.h < 0.f;
  }
  return cnt;
}
// multisect_eigs with the Sturm counts in double-float (FP32 pipes): the
// intervals stop at ~2^-44 of ||T|| (atol) or 2^-45 relative.  Meant for all the
// warps of a CTA at once (t0 = warp, tstride = warps), so each eigenvalue gets
// several lanes and rounds are few.
__device__ inline void multisect_eigs_df(const dfl* d, const dfl* e2, int n, int k, int t0, int tstride,
                                         double lo0, double hi0, float pivmin, double atol, double wscale, double* w) {
  const int lane = threadIdx.x & 31;
  const int ng = (k - t0 + tstride - 1) / tstride;          // eigenvalues of this warp
  if (ng <= 0) return;
  const int L = max(1, 32 / ng);
  const int gmax = 32 / L;
  const double eps = 2.842170943040401e-14;                 // 2^-45
  for (int gb = 0; gb < ng; gb += gmax) {
    const int g = gb + lane / L, q = lane % L;
    const int t = t0 + g * tstride;
    const bool mine = (lane / L < gmax) && (g < ng) && (t < k);
    const int j = n - 1 - t;
    double lo = lo0, hi = hi0;
    bool done = !mine;
    for (int it = 0; it < 200; it++) {
      if (!__any_sync(0xffffffffu, !done)) break;
      const double x = lo + (hi - lo) * (double)(q + 1) / (double)(L + 1);
      bool above = false;
      if (!done) above = sturm_count_df(d, e2, n, x, pivmin) > j;
      const unsigned bal = __ballot_sync(0xffffffffu, above);
      if (!done) {
        const unsigned bits = (bal >> ((lane / L) * L)) & ((L == 32) ? 0xffffffffu : ((1u << L) - 1u));
        const int qs = bits ? (__ffs(bits) - 1) : L;
        const double nlo = (qs == 0) ? lo : lo + (hi - lo) * (double)qs / (double)(L + 1);
        const double nhi = (qs == L) ? hi : lo + (hi - lo) * (double)(qs + 1) / (double)(L + 1);
        if (!(nlo > lo || nhi < hi)) done = true;
        lo = nlo;
        hi = nhi;
        if (hi - lo <= fmax(2.0 * eps * fmax(fabs(lo), fabs(hi)), atol)) done = true;
      }
    }
    if (mine && q == 0) w[t] = 0.5 * (lo + hi) * wscale;
  }
  __syncwarp();
}

// (T - lam I) x = y by Gaussian elimination with partial pivoting on the tridiagonal, for many
// shifts at once, one per lane of a warp: element i of a lane's arrays at [i * 32] from the lane's base pointer,
// so a warp's accesses are coalesced.  Branch-free, one division per row
// (the inverse pivot ui = 1 / u0 is kept), so the lanes do not diverge.
__device__ inline void tri_factor_lanes(const double* d, const double* e, int n, double lam, double small,
                                        double* ui, double* u1, double* u2, double* mul, int* piv) {
  double wa = d[0] - lam, wb = (n > 1) ? e[0] : 0.0;
  for (int i = 0; i + 1 < n; i++) {
    const double c = e[i], a1 = d[i + 1] - lam, b1 = (i + 2 < n) ? e[i + 1] : 0.0;
    const bool keep = fabs(wa) >= fabs(c);
    const double a = keep ? (wa == 0.0 ? small : wa) : c;
    const double inv = 1.0 / a;
    const double m = (keep ? c : wa) * inv;
    ui[32 * i] = inv;
    u1[32 * i] = keep ? wb : a1;
    u2[32 * i] = keep ? 0.0 : b1;
    mul[32 * i] = m;
    piv[32 * i] = keep ? 0 : 1;
    const double na = keep ? a1 - m * wb : wb - m * a1;
    wb = keep ? b1 : -m * b1;
    wa = na;
  }
  ui[32 * (n - 1)] = 1.0 / ((wa == 0.0) ? small : wa);
  u1[32 * (n - 1)] = 0.0;
  u2[32 * (n - 1)] = 0.0;
}
// y <- (T - lam I)^{-1} (sc y) for each lane's vector, returning |x|^2 of the
// result.  The element loads of each sweep are issued eight rows ahead of the
// recurrence (the arrays live in L2), so their latency is not paid per row.
__device__ inline double tri_solve_lanes(int n, double sc, const double* ui, const double* u1, const double* u2,
                                         const double* mul, const int* piv, double* y) {
  constexpr int U = 8;
  double cur = sc * y[0];
  int i = 0;
  for (; i + U < n; i += U) {
    double nx[U], mu[U];
    int pv[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      nx[u] = y[32 * (i + 1 + u)];
      mu[u] = mul[32 * (i + u)];
      pv[u] = piv[32 * (i + u)];
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      const double v = sc * nx[u];
      const bool sw = pv[u] != 0;
      const double lo = sw ? v : cur, hi = sw ? cur : v;
      y[32 * (i + u)] = lo;
      cur = hi - mu[u] * lo;
    }
  }
  for (; i + 1 < n; i++) {
    const double v = sc * y[32 * (i + 1)];
    const bool sw = piv[32 * i] != 0;
    const double lo = sw ? v : cur, hi = sw ? cur : v;
    y[32 * i] = lo;
    cur = hi - mul[32 * i] * lo;
  }
  y[32 * (n - 1)] = cur;
  double y1 = 0.0, y2 = 0.0, nn = 0.0;   // x[i + 1], x[i + 2]
  i = n - 1;
  for (; i - U + 1 >= 0; i -= U) {
    double yv[U], a1[U], a2[U], iv[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      yv[u] = y[32 * (i - u)];
      a1[u] = u1[32 * (i - u)];
      a2[u] = u2[32 * (i - u)];
      iv[u] = ui[32 * (i - u)];
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      const double x = (yv[u] - a1[u] * y1 - a2[u] * y2) * iv[u];
      y[32 * (i - u)] = x;
      nn += x * x;
      y2 = y1;
      y1 = x;
    }
  }
  for (; i >= 0; i--) {
    const double x = (y[32 * i] - u1[32 * i] * y1 - u2[32 * i] * y2) * ui[32 * i];
    y[32 * i] = x;
    nn += x * x;
    y2 = y1;
    y1 = x;
  }
  return nn;
}

// 1/a in double-float: the rounded FP32 reciprocal refined by one Newton step
// (the residual 1 - a_h r is exact in an FMA), ~47 bits.
__device__ __forceinline__ dfl df_rcp(dfl a) {
  const float r = 1.0f / a.h;
  float e = fmaf(-a.h, r, 1.0f);
  e = fmaf(-a.l, r, e);
  return df_fast2(r, r * e);
}
// tri_factor_lanes in double-float arithmetic (the mixed-form OSV build): d and e
// as (hi, lo) pairs, the factors stored as pairs in the same lane-interleaved
// slots, so the recurrence runs on the FP32 pipes.
__device__ inline void tri_factor_lanes_df(const dfl* d, const dfl* e, int n, dfl lam, float small, dfl* ui,
                                           dfl* u1, dfl* u2, dfl* mul, int* piv) {
  const dfl z{0.f, 0.f}, nl = df_neg(lam);
  dfl wa = df_add(d[0], nl), wb = (n > 1) ? e[0] : z;
  for (int i = 0; i + 1 < n; i++) {
    const dfl c = e[i], a1 = df_add(d[i + 1], nl), b1 = (i + 2 < n) ? e[i + 1] : z;
    const bool keep = fabsf(wa.h) >= fabsf(c.h);
    const dfl a = keep ? (wa.h == 0.f ? dfl{small, 0.f} : wa) : c;
    const dfl inv = df_rcp(a);
    const dfl m = df_mul(keep ? c : wa, inv);
    ui[32 * i] = inv;
    u1[32 * i] = keep ? wb : a1;
    u2[32 * i] = keep ? z : b1;
    mul[32 * i] = m;
    piv[32 * i] = keep ? 0 : 1;
    const dfl nm = df_neg(m);
    const dfl na = keep ? df_fma1(nm, wb, a1) : df_fma1(nm, a1, wb);
    wb = keep ? b1 : df_mul(nm, b1);
    wa = na;
  }
  ui[32 * (n - 1)] = df_rcp(wa.h == 0.f ? dfl{small, 0.f} : wa);
  u1[32 * (n - 1)] = z;
  u2[32 * (n - 1)] = z;
}
// tri_solve_lanes in double-float: y <- (T - lam I)^{-1} (sc y), returning max |x|
// (the next solve's scale; the vectors are normalised in FP64 afterwards).
__device__ inline float tri_solve_lanes_df(int n, float sc, const dfl* ui, const dfl* u1, const dfl* u2,
                                           const dfl* mul, const int* piv, dfl* y) {
  constexpr int U = 4;
  const dfl s{sc, 0.f};
  dfl cur = df_mul(y[0], s);
  int i = 0;
  for (; i + U < n; i += U) {
    dfl nx[U], mu[U];
    int pv[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      nx[u] = y[32 * (i + 1 + u)];
      mu[u] = mul[32 * (i + u)];
      pv[u] = piv[32 * (i + u)];
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      const dfl v = df_mul(nx[u], s);
      const bool sw = pv[u] != 0;
      const dfl lo = sw ? v : cur, hi = sw ? cur : v;
      y[32 * (i + u)] = lo;
      cur = df_fma1(df_neg(mu[u]), lo, hi);
    }
  }
  for (; i + 1 < n; i++) {
    const dfl v = df_mul(y[32 * (i + 1)], s);
    const bool sw = piv[32 * i] != 0;
    const dfl lo = sw ? v : cur, hi = sw ? cur : v;
    y[32 * i] = lo;
    cur = df_fma1(df_neg(mul[32 * i]), lo, hi);
  }
  y[32 * (n - 1)] = cur;
  const dfl z{0.f, 0.f};
  dfl y1 = z, y2 = z;   // x[i + 1], x[i + 2]
  float amax = 0.f;
  i = n - 1;
  for (; i - U + 1 >= 0; i -= U) {
    dfl yv[U], a1[U], a2[U], iv[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      yv[u] = y[32 * (i - u)];
      a1[u] = u1[32 * (i - u)];
      a2[u] = u2[32 * (i - u)];
      iv[u] = ui[32 * (i - u)];
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      const dfl x = df_mul(df_fma2(df_neg(a1[u]), y1, df_neg(a2[u]), y2, yv[u]), iv[u]);
      y[32 * (i - u)] = x;
      amax = fmaxf(amax, fabsf(x.h));
      y2 = y1;
      y1 = x;
    }
  }
  for (; i >= 0; i--) {
    const dfl x = df_mul(df_fma2(df_neg(u1[32 * i]), y1, df_neg(u2[32 * i]), y2, y[32 * i]), ui[32 * i]);
    y[32 * i] = x;
    amax = fmaxf(amax, fabsf(x.h));
    y2 = y1;
    y1 = x;
  }
  return amax;
}

}  // namespace osv

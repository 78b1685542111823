// A3 of both forms (the FP64 form skips the leftovers and polishes the basis afterwards,
// solve_oz.cu): a basis X of the pair space with X^T F X ~ diag(e~) and
// X^T S X ~ 1 (Eq. prec_eig), plus the exact leftovers
//   S^ = X^T S X - 1,   G^ = (X^T F X - diag(e~)) - (f_ii + f_jj)/2 S^
// (double-float products, stored FP32: they are ~1e-7) that the mixed fragment solver
// adds to its update, so the iteration's fixed point is the exact one whatever
// the accuracy of X.
//
// Canonical orthogonalisation through the block structure of the overlap:
// S_(ij,ij) = [[1, M], [M^T, 1]] with M = Q_i^T Q_j (the OSVs of each orbital
// are orthonormal).  With C = 1 - M^T M = V diag(mu) V^T (FP64, order n_j),
//   Y = [[1, -M Z], [0, Z]],  Z = V_kept diag(mu_kept)^(-1/2),
// gives Y^T S Y = blockdiag(1, Z^T C Z) = 1.  The eigenvalues of S are 1 and
// 1 +- sigma_k (sigma_k^2 = 1 - mu_k), and a direction is dropped exactly when
// the canonical orthogonalisation drops the eigenvalue 1 - sigma_k =
// mu_k / (1 + sigma_k) below tau_s (1 + sigma_max).  Then F' = Y^T F Y (double-float,
// entries bounded by the virtual energies whatever the conditioning of Y) is
// diagonalised in FP32 (F' = W diag(e~) W^T) and X = Y W.  A diagonal pair has
// S_(ii,ii) = Q_i^T Q_i = 1: Y = 1, F' = F_(i,i).
//
// Launches (CTA kernels take one pair per CTA, grid-stride over the pairs in
// descending order, so the largest start first):
//   (0)  Y by Cholesky wherever no direction is dropped (or all are); the other pairs:
//   (1a) C = 1 - M^T M, Householder tridiagonalisation and Z (FP64, CTA);
//   (1b) the QR bulge chase of every C, one pair per thread (FP64);
//   (1c) recorded rotations applied to Z, kept directions, Y, Z^T C Z (CTA; the
//        products with Z in double-float);
//   (2)  F' = Y^T F Y (tiled double-float GEMMs, CTA);
//   (3)  F' diagonalised by FP32 Jacobi rotations; (3a-c) the three steps for orders beyond its
//        shared memory;
//   (4)  X = Y W and the leftovers (tiled double-float GEMMs, CTA).
// C and its eigen-decomposition stay FP64: C = 1 - M^T M cancels, and its small
// eigenvalues set both the kept directions and Z.  The products with Z, Y and W
// carry ~2^-48 relative error; it enters X, U = P X and the leftovers alike, so
// the fixed point does not move.
// The eigen-solver is Householder + implicit QR (eig.cuh) with the chase run
// per thread over many pairs at once and its rotations recorded, then applied
// to the eigenvectors (kept column-major, so the rotations are coalesced) by a
// CTA; a pair whose record overflows is redone by the in-CTA solver.
// Per-pair intermediates live in a scratch slot: Y [m][r], F' [r][r], W [r][r],
// Z^T C Z [nk][nk], e~ [r], and the eigen-solver's work area.
#include <algorithm>

#include "eig.cuh"
#include "pairview.cuh"

namespace osv {


// eigen-solver work area of a pair of order m: status and sweep count, Z (m x m),
// d and e (m each), the sweep record (cap_s (l, h) pairs) and the rotation
// record (cap_r (c, s) pairs); typed FP64 or FP32 by the step that uses it
__host__ __device__ inline int pm_cap_s(int m) { return 4 * m + 64; }
__host__ __device__ inline int pm_cap_r(int m) { return 2 * m * m + 64; }
__host__ __device__ inline size_t pm_work_doubles(int m) {
  return 2 + (size_t)m * m + 2 * (size_t)m + (size_t)pm_cap_s(m) + 2 * (size_t)pm_cap_r(m);
}
__host__ __device__ inline size_t pm_slot_doubles(int m) {
  return 4 * (size_t)m * m + (size_t)m + 8 + pm_work_doubles(m);
}
// per-CTA scratch: (1) C, C0, V [3][max_m^2] + mu, e, tau; (2) F Y; (3) FP32 A, Z, e~, e, tau; (4) 3 blocks
__host__ __device__ inline size_t pm_cta_doubles(int max_m) {
  return 3 * (size_t)max_m * max_m + 3 * (size_t)max_m;
}

struct PmPair {              // per-pair view of the scratch slot
  double* Y;                 // [m][r]
  double* Fp;                // [r][r]
  double* W;                 // [r][r]
  double* ZCZ;               // [nk][nk]
  double* et;                // [r]
  double* wk;                // eigen-solver work area
};
__device__ __forceinline__ PmPair pm_pair(double* slots, const long long* off, int jid, int m) {
  double* b = slots + off[jid];
  const size_t M2 = (size_t)m * m;
  return PmPair{b, b + M2, b + 2 * M2, b + 3 * M2, b + 4 * M2, b + 4 * M2 + m + 8};
}

template <class T>
struct PmEig {               // typed view of a pair's eigen-solver work area
  int* hdr;                  // [0] status of the chase (0, 1 no convergence, 2 record overflow), [1] sweeps,
                             // [2] Y formed by k_pm_chol, [3] F' diagonalised by k_pm_jacobi
  T* Z;                      // eigenvector t at Z[t * n ..] (column-major eigenvector matrix)
  T* d;                      // eigenvalues after the chase
  T* e;
  int* swp;
  T* rot;
};
template <class T>
__device__ __forceinline__ PmEig<T> pm_eig(double* wk, int m) {
  const size_t M2 = (size_t)m * m;
  PmEig<T> w;
  w.hdr = reinterpret_cast<int*>(wk);
  w.Z = reinterpret_cast<T*>(wk + 2);
  w.d = reinterpret_cast<T*>(wk + 2 + M2);
  w.e = reinterpret_cast<T*>(wk + 2 + M2 + m);
  w.swp = reinterpret_cast<int*>(wk + 2 + M2 + 2 * m);
  w.rot = reinterpret_cast<T*>(wk + 2 + M2 + 2 * m + pm_cap_s(m));
  return w;
}

// Householder tridiagonalisation of A (order n, destroyed) and the column-major
// Z of its reflectors into the work area (CTA); tau: n elements, sm: 4n + 33.
template <class T>
__device__ void pm_tridiag(T* A, int n, const PmEig<T>& w, T* tau, T* sm) {
  if (n == 1) {
    if (threadIdx.x == 0) { w.d[0] = A[0]; w.e[0] = T(0.0); w.Z[0] = T(1.0); }
    __syncthreads();
    return;
  }
  cta_tridiag(A, n, n, w.d, w.e, tau, sm, sm + n, sm + 4 * n);
  cta_form_z_cm(A, n, n, tau, w.Z, n, sm, sm + n);
  if (threadIdx.x == 0) w.e[n - 1] = T(0.0);
  __syncthreads();
}

// (1b) / (3b): the QR chase of one pair per lane; which = 0: C (order n_j), 1: F' (order r).  Pairs in the order
// array, so a warp holds pairs of similar size; lpw lanes of a warp have one each (as few as the number of pairs
// allows with a warp on every SM sub-partition: a serial chain gains nothing from sharing its warp, and every lane
// adds the divergence of its own sweeps).  Orders up to nsm run on copies of d and e in shared memory, interleaved
// by lane (they are read and written at every rotation).  Dynamic shared memory: 2 nsm 32 elements.
template <class T>
__global__ void __launch_bounds__(32) k_pm_chase(Tables t, const PJob* __restrict__ jobs,
                                                 const int* __restrict__ order, int n_jobs, double* slots,
                                                 const long long* off, const int* mdim, int which, int lpw, int nsm,
                                                 int* err) {
  extern __shared__ double chase_raw[];
  T* sh = reinterpret_cast<T*>(chase_raw);
  const int lane = threadIdx.x, q = blockIdx.x * lpw + lane;
  if (lane >= lpw || q >= n_jobs) return;
  const int jid = order[q];
  const PJob jb = jobs[jid];
  const int m = mdim[jid];
  const int ne = which == 0 ? (jb.i == jb.j ? 0 : t.n_osv[jb.j]) : *jb.r;
  if (ne == 0) return;
  const PmEig<T> w = pm_eig<T>(pm_pair(slots, off, jid, m).wk, m);
  if (w.hdr[which == 0 ? 2 : 3]) return;
  int ns = 0, rc;
  if (ne <= nsm) {
    T *d = sh + lane, *e = sh + (size_t)32 * nsm + lane;
    for (int k = 0; k < ne; k++) {
      d[32 * k] = w.d[k];
      e[32 * k] = w.e[k];
    }
    rc = tridiag_qr_record<32>(d, e, ne, w.swp, pm_cap_s(m), w.rot, pm_cap_r(m), &ns);
    for (int k = 0; k < ne; k++) w.d[k] = d[32 * k];
  } else {
    rc = tridiag_qr_record(w.d, w.e, ne, w.swp, pm_cap_s(m), w.rot, pm_cap_r(m), &ns);
  }
  w.hdr[0] = rc;
  w.hdr[1] = ns;
  if (rc == 1) atomicOr(err, ERR_EIG);
}

// (0) Y of the pairs whose space is clearly not dependent: with C = 1 - M^T M = L L^T (FP64 Cholesky in shared
// memory) any Z with Z^T C Z = 1 serves, here Z = L^(-T), provided that no direction is to be dropped.  That
// is certain when trace(C^-1) = |L^-1|_F^2 < 1 / (4 tau_s): the smallest eigenvalue of C is at least
// 1 / trace(C^-1), and a direction is dropped only if mu_k / (1 + sqrt(1 - mu_k)) <= tau_s smax with smax <= 2.
// When |C|_F <= tau_s every direction is dropped (mu_k <= |C|_F, smax >= 1).  All other pairs keep hdr[2] = 0
// and go through the eigen-decomposition of C below.  One CTA per pair; the eigen-decomposition's tridiagonalisation,
// one-thread QR chase and rotations took 21 ms at 128 orbitals (1584 pairs of ~46 + 46 OSVs), this 5.2 ms.
// Dynamic shared memory: nmax (nmax + 1) + nmax doubles.
__global__ void __launch_bounds__(NT) k_pm_chol(Tables t, double tau_s, const PJob* __restrict__ jobs,
                                                const int* __restrict__ order, int n_jobs, double* slots,
                                                const long long* off, int max_m, int nmax, double* scratch) {
  __shared__ double gsm[GEMM_SMEM_DOUBLES];
  __shared__ double red[40];
  extern __shared__ double cs[];
  __shared__ int s_bad;
  const size_t M2 = (size_t)max_m * max_m;
  double* C0 = scratch + (size_t)blockIdx.x * pm_cta_doubles(max_m);
  double* CZ = C0 + M2;
  const int n = t.n_occ, tid = threadIdx.x;
  for (int q = blockIdx.x; q < n_jobs; q += gridDim.x) {
    const int jid = order[q];
    const PJob jb = jobs[jid];
    const int i = jb.i, j = jb.j;
    const int ni = t.n_osv[i], nj = (i == j) ? 0 : t.n_osv[j], m = ni + nj;
    const PmPair pp = pm_pair(slots, off, jid, m);
    int* hdr = pm_eig<double>(pp.wk, m).hdr;
    if (tid == 0) {
      hdr[2] = hdr[3] = 0;
      s_bad = 0;
      if (i == j) *jb.r = ni;
    }
    __syncthreads();
    if (i == j || nj > nmax) continue;
    const int ld = nj | 1;
    double* dinv = cs + (size_t)nmax * (nmax + 1);
    const View Mv = dense_view(t.S[t.sf_id[i * n + j]], ni, nj, nj);
    cta_gemm(nj, nj, ni, -1.0, transpose(Mv), Mv, 0.0, cs, ld, gsm);
    double fro = 0.0;
    for (int idx = tid; idx < nj * nj; idx += NT) {
      const int a = idx / nj, b = idx % nj;
      const double c = cs[(size_t)a * ld + b] + (a == b ? 1.0 : 0.0);
      cs[(size_t)a * ld + b] = c;
      C0[idx] = c;
      fro += c * c;
    }
    fro = cta_sum(fro, red);
    int nk = nj;
    if (fro <= tau_s * tau_s) nk = 0;
    else {
      // C = L L^T in the lower triangle, 1 / L_kk in dinv
      for (int k = 0; k < nj; k++) {
        const double p = cs[(size_t)k * ld + k];
        if (!(p > 0.0)) {          // the same in every thread
          if (tid == 0) s_bad = 1;
          break;
        }
        const double inv = 1.0 / sqrt(p);
        if (tid == 0) dinv[k] = inv;
        __syncthreads();
        for (int a = k + 1 + tid; a < nj; a += NT) cs[(size_t)a * ld + k] *= inv;
        __syncthreads();
        const int L = nj - k - 1;
        for (int idx = tid; idx < L * L; idx += NT) {
          const int a = k + 1 + idx / L, b = k + 1 + idx % L;
          if (b <= a) cs[(size_t)a * ld + b] = fma(-cs[(size_t)a * ld + k], cs[(size_t)b * ld + k], cs[(size_t)a * ld + b]);
        }
        __syncthreads();
      }
      __syncthreads();
      const int bad = s_bad;
      __syncthreads();
      if (bad) continue;
      // rows of Z = L^(-T) (row c: column c of L^-1) in the upper triangle, the diagonal in dinv
      double tr = 0.0;
      for (int c = tid; c < nj; c += NT) {
        const double d = dinv[c];
        double* z = cs + (size_t)c * ld;
        tr += d * d;
        for (int a = c + 1; a < nj; a++) {
          const double* La = cs + (size_t)a * ld;
          double s0 = La[c] * d, s1 = 0.0, s2 = 0.0, s3 = 0.0;
          int k = c + 1;
          for (; k + 3 < a; k += 4) {
            s0 = fma(La[k], z[k], s0);
            s1 = fma(La[k + 1], z[k + 1], s1);
            s2 = fma(La[k + 2], z[k + 2], s2);
            s3 = fma(La[k + 3], z[k + 3], s3);
          }
          for (; k < a; k++) s0 = fma(La[k], z[k], s0);
          const double x = -dinv[a] * ((s0 + s1) + (s2 + s3));
          z[a] = x;
          tr += x * x;
        }
      }
      tr = cta_sum(tr, red);
      if (!(tr * 4.0 * tau_s < 1.0)) continue;
    }
    const int r = ni + nk;
    double* Y = pp.Y;
    for (int idx = tid; idx < m * r; idx += NT) {
      const int a = idx / r, b = idx % r;
      double y = 0.0;
      if (a < ni) y = (b == a) ? 1.0 : 0.0;
      else if (b >= ni) {
        const int za = a - ni, zb = b - ni;
        y = za == zb ? dinv[za] : (za < zb ? cs[(size_t)za * ld + zb] : 0.0);
      }
      Y[idx] = y;
    }
    __syncthreads();
    const View Zv = dense_view(Y + (size_t)ni * r + ni, nj, nk, r);
    cta_gemm_df_r<4>(ni, nk, nj, -1.0, Mv, Zv, 0.0, Y + ni, r, gsm);                                     // -M Z
    if (jb.Sh) {                                                                                         // leftovers
      cta_gemm_df_r<4>(nj, nk, nj, 1.0, dense_view(C0, nj, nj, nj), Zv, 0.0, CZ, nk, gsm);                // C Z
      cta_gemm_df_r<4>(nk, nk, nj, 1.0, transpose(Zv), dense_view(CZ, nj, nk, nk), 0.0, pp.ZCZ, nk, gsm);  // Z^T C Z
    }
    if (tid == 0) {
      *jb.r = r;
      hdr[2] = 1;
    }
    __syncthreads();
  }
}

// (3) F' diagonalised in FP32 by cyclic Jacobi with the rotations of a round in parallel (round-robin
// pairing: r / 2 disjoint rotations, r - 1 rounds a sweep), A (upper triangle) and the rows of V^T in shared
// memory.  A round is two barriers, ~r^2 / 8 blocks of 2 x 2 of A and r^2 / 2 pairs of V elements; a warp takes a
// row of blocks (rows i and np - 1 - i of the triangle together) and a row pair of V, so that no lane divides and
// neighbouring lanes meet neighbouring banks (odd row stride).  Issue-bound (5.9k instructions a round at order 90,
// 2.2 a clock; 8 sweeps).  With few pairs the Householder reduction, one-lane chase and rotation replay of the steps
// below spend most of their time in serial steps (32 orbitals, 300 pairs: ~5 ms against 2.7 here); with many pairs
// they hide it and need fewer operations, so launch_precond_mixed chooses.  The leftovers or the polish take up the
// rounding errors of the vectors.  Orders above jmax (two matrices in shared memory) go through the steps below too.
constexpr int NT_J = 512;
__global__ void __launch_bounds__(NT_J) k_pm_jacobi(const PJob* __restrict__ jobs, const int* __restrict__ order,
                                                    int n_jobs, double* slots, const long long* off, const int* mdim,
                                                    int jmax, int* err) {
  extern __shared__ float js[];
  __shared__ float2 cs[128];
  __shared__ short2 pq[128];           // p < q; q = -1: the odd one out rests
  __shared__ float redf[33];
  __shared__ int s_any;
  constexpr int NW = NT_J / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int jq = blockIdx.x; jq < n_jobs; jq += gridDim.x) {
    const int jid = order[jq];
    const PJob jb = jobs[jid];
    const int m = mdim[jid], r = *jb.r;
    const PmPair pp = pm_pair(slots, off, jid, m);
    if (r > jmax || r < 1) continue;
    const int ld = r | 1;
    float* A = js;                       // upper triangle, A[p * ld + q], p <= q
    float* V = js + (size_t)r * ld;      // V[k * ld + a]: component a of vector k
    float amax = 0.f;
    bool bad = false;
    for (int idx = tid; idx < r * r; idx += NT_J) {
      const int a = idx / r, b = idx % r;
      const float x = (float)(0.5 * (pp.Fp[idx] + pp.Fp[(size_t)b * r + a]));
      A[a * ld + b] = x;
      V[a * ld + b] = a == b ? 1.f : 0.f;
      amax = fmaxf(amax, fabsf(x));
      bad |= !isfinite(x);
    }
    bad = __syncthreads_or(bad);
    if (bad) {
      if (tid == 0) atomicOr(err, ERR_NONFINITE);
      __syncthreads();
      continue;
    }
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if (lane == 0) redf[warp] = amax;
    __syncthreads();
    if (tid == 0) {
      for (int k = 1; k < NW; k++) amax = fmaxf(amax, redf[k]);
      redf[32] = amax;
      s_any = 0;
    }
    __syncthreads();
    const float tiny = 6e-8f * redf[32];   // an FP32 ulp of the largest entry: nothing left to rotate
    const int n2 = r + (r & 1), np = n2 / 2, n1 = n2 - 1;
    int sweep = 0;
    for (; sweep < 16; sweep++) {
      for (int rd = 0; rd < n1; rd++) {
        if (tid < np) {
          int p = rd + tid, q = rd - tid;
          if (p >= n1) p -= n1;
          if (q < 0) q += n1;
          if (tid == 0) p = n1;
          if (p > q) { const int x = p; p = q; q = x; }
          float c = 1.f, s = 0.f;
          if (q < r) {
            const float x = A[p * ld + q];
            if (fabsf(x) > tiny) {
              const float th = (A[q * ld + q] - A[p * ld + p]) / (2.f * x);
              const float tt = copysignf(1.f, th) / (fabsf(th) + sqrtf(1.f + th * th));
              c = 1.f / sqrtf(1.f + tt * tt);
              s = tt * c;
              s_any = 1;
            }
          } else q = -1;
          pq[tid] = make_short2((short)p, (short)q);
          cs[tid] = make_float2(c, s);
        }
        __syncthreads();
        // A <- J^T A J by 2 x 2 blocks (i, j), i <= j; new row p = c row p - s row q, row q = s row p + c row q
        for (int w = warp; 2 * w < np; w += NW)
          for (int u0 = lane; u0 <= np; u0 += 32) {
            // rows w and np - 1 - w of the triangle hold np - w and w + 1 blocks
            int i = w, j = w + u0;
            if (u0 >= np - w) {
              i = np - 1 - w;
              j = i + (u0 - (np - w));
              if (i == w) break;         // the middle row of an odd count stands alone
            }
            const short2 P = pq[i], U = pq[j];
            const float2 ci = cs[i], cj = cs[j];
            const int p = P.x, q = P.y, u = U.x, v = U.y;
            const float c = ci.x, s = ci.y, c2 = cj.x, s2 = cj.y;
            if (i == j) {
              if (s == 0.f) continue;
              const float app = A[p * ld + p], apq = A[p * ld + q], aqq = A[q * ld + q];
              const float r0 = c * app - s * apq, r1 = c * apq - s * aqq, t0 = s * app + c * apq, t1 = s * apq + c * aqq;
              A[p * ld + p] = c * r0 - s * r1;
              A[p * ld + q] = 0.f;
              A[q * ld + q] = s * t0 + c * t1;
              continue;
            }
            if (s == 0.f && s2 == 0.f) continue;
            float* e00 = A + (p < u ? p * ld + u : u * ld + p);
            if (q >= 0 && v >= 0) {
              float* e01 = A + (p < v ? p * ld + v : v * ld + p);
              float* e10 = A + (q < u ? q * ld + u : u * ld + q);
              float* e11 = A + (q < v ? q * ld + v : v * ld + q);
              const float v00 = *e00, v01 = *e01, v10 = *e10, v11 = *e11;
              const float a0 = c * v00 - s * v10, a1 = c * v01 - s * v11, b0 = s * v00 + c * v10, b1 = s * v01 + c * v11;
              *e00 = c2 * a0 - s2 * a1;
              *e01 = s2 * a0 + c2 * a1;
              *e10 = c2 * b0 - s2 * b1;
              *e11 = s2 * b0 + c2 * b1;
            } else if (v >= 0) {         // row p alone
              float* e01 = A + (p < v ? p * ld + v : v * ld + p);
              const float v00 = *e00, v01 = *e01;
              *e00 = c2 * v00 - s2 * v01;
              *e01 = s2 * v00 + c2 * v01;
            } else {                     // column u alone
              float* e10 = A + (q < u ? q * ld + u : u * ld + q);
              const float v00 = *e00, v10 = *e10;
              *e00 = c * v00 - s * v10;
              *e10 = s * v00 + c * v10;
            }
          }
        for (int i = warp; i < np; i += NW) {
          const float2 ci = cs[i];
          if (ci.y == 0.f) continue;
          const short2 P = pq[i];
          const float tau = ci.y / (1.f + ci.x);   // c = 1 - s tau: no rounding of c enters the norms
          float *x = V + P.x * ld, *y = V + P.y * ld;
          for (int a = lane; a < r; a += 32) {
            const float vx = x[a], vy = y[a];
            x[a] = fmaf(-ci.y, fmaf(tau, vx, vy), vx);
            y[a] = fmaf(ci.y, fmaf(-tau, vy, vx), vy);
          }
        }
        __syncthreads();
      }
      const int any = s_any;
      __syncthreads();
      if (!any) break;
      if (tid == 0) s_any = 0;
      __syncthreads();
    }
    for (int idx = tid; idx < r * r; idx += NT_J) {   // W[a][k] = component a of vector k
      const int a = idx / r, k = idx % r;
      pp.W[idx] = (double)V[k * ld + a];
    }
    for (int k = tid; k < r; k += NT_J) pp.et[k] = (double)A[k * ld + k];
    if (tid == 0) pm_eig<double>(pp.wk, m).hdr[3] = sweep < 16;   // not converged: the steps below take it
    __syncthreads();
  }
}

// (1a) C = 1 - M^T M, tridiagonalised, Z of the reflectors
__global__ void __launch_bounds__(NT, 3) k_pm_overlap_a(Tables t, const PJob* __restrict__ jobs,
                                                        const int* __restrict__ order, int n_jobs, double* slots,
                                                        const long long* off, int max_m, double* scratch) {
  __shared__ double gsm[GEMM_SMEM_DOUBLES];
  extern __shared__ double esm[];   // eigen-solver scratch: 4 max_m + 33 doubles
  const size_t M2 = (size_t)max_m * max_m;
  double* Cw = scratch + (size_t)blockIdx.x * pm_cta_doubles(max_m);
  double* tau = Cw + M2;
  const int n = t.n_occ;
  for (int q = blockIdx.x; q < n_jobs; q += gridDim.x) {
    const int jid = order[q];
    const PJob jb = jobs[jid];
    const int i = jb.i, j = jb.j;
    if (i == j) continue;
    const int ni = t.n_osv[i], nj = t.n_osv[j], m = ni + nj;
    if (pm_eig<double>(pm_pair(slots, off, jid, m).wk, m).hdr[2]) continue;
    const View Mv = dense_view(t.S[t.sf_id[i * n + j]], ni, nj, nj);
    cta_gemm(nj, nj, ni, -1.0, transpose(Mv), Mv, 0.0, Cw, nj, gsm);
    for (int c = threadIdx.x; c < nj; c += NT) Cw[(size_t)c * nj + c] += 1.0;
    __syncthreads();
    pm_tridiag(Cw, nj, pm_eig<double>(pm_pair(slots, off, jid, m).wk, m), tau, esm);
  }
}

// (1c) eig(C) completed (mu, V), kept directions, Y, Z^T C Z, r
__global__ void __launch_bounds__(NT, 3) k_pm_overlap_c(Tables t, double tau_s, const PJob* __restrict__ jobs,
                                                        const int* __restrict__ order, int n_jobs, double* slots,
                                                        const long long* off, int max_m, double* scratch,
                                                        int* err) {
  __shared__ double gsm[GEMM_SMEM_DOUBLES];
  extern __shared__ double esm[];   // eigen-solver scratch: 4 max_m + 33 doubles, then keep [max_m]
  int* keep = reinterpret_cast<int*>(esm + 4 * max_m + 33);
  __shared__ int s_nk;
  const size_t M2 = (size_t)max_m * max_m;
  double* C0 = scratch + (size_t)blockIdx.x * pm_cta_doubles(max_m);
  double* CZ = C0 + M2;
  double* Af = CZ + M2;         // in-CTA solve of a pair whose chase record overflowed
  double* muf = Af + M2;
  double* ef = muf + max_m;
  double* tauf = ef + max_m;
  const int n = t.n_occ;
  for (int q = blockIdx.x; q < n_jobs; q += gridDim.x) {
    const int jid = order[q];
    const PJob jb = jobs[jid];
    const int i = jb.i, j = jb.j;
    const int ni = t.n_osv[i], nj = (i == j) ? 0 : t.n_osv[j];
    const int m = ni + nj;
    const PmPair pp = pm_pair(slots, off, jid, m);
    if (i == j || pm_eig<double>(pp.wk, m).hdr[2]) continue;
    const View Mv = dense_view(t.S[t.sf_id[i * n + j]], ni, nj, nj);
    cta_gemm(nj, nj, ni, -1.0, transpose(Mv), Mv, 0.0, C0, nj, gsm);
    for (int c = threadIdx.x; c < nj; c += NT) C0[(size_t)c * nj + c] += 1.0;
    __syncthreads();
    const PmEig<double> w = pm_eig<double>(pp.wk, m);
    const double* mu = w.d;
    const double* V = w.Z;      // eigenvector k of C at V[k * nj ..]
    if (w.hdr[0] == 2) {
      for (int idx = threadIdx.x; idx < nj * nj; idx += NT) Af[idx] = C0[idx];
      __syncthreads();
      if (cta_syev_cm(Af, nj, nj, muf, w.Z, nj, ef, tauf, esm) && threadIdx.x == 0) atomicOr(err, ERR_EIG);
      mu = muf;
    } else {
      apply_qr_record_cm(w.Z, nj, nj, w.swp, w.hdr[1], w.rot);
    }
    if (threadIdx.x == 0) {
      double mumin = 1.0;
      for (int k = 0; k < nj; k++) mumin = fmin(mumin, mu[k]);
      const double smax = 1.0 + sqrt(fmax(0.0, 1.0 - mumin));
      int nk = 0;
      for (int k = 0; k < nj; k++) {
        const double lam = mu[k] / (1.0 + sqrt(fmax(0.0, 1.0 - mu[k])));
        if (mu[k] > 0.0 && lam > tau_s * smax) keep[nk++] = k;
      }
      s_nk = nk;
    }
    __syncthreads();
    const int nk = s_nk, r = ni + nk;
    double* Y = pp.Y;
    for (int idx = threadIdx.x; idx < m * r; idx += NT) {
      const int a = idx / r, b = idx % r;
      double y = 0.0;
      if (a < ni) y = (b == a) ? 1.0 : 0.0;
      else if (b >= ni) {
        const int k = keep[b - ni];
        y = V[(size_t)k * nj + (a - ni)] / sqrt(mu[k]);
      }
      Y[idx] = y;
    }
    __syncthreads();
    const View Zv = dense_view(Y + (size_t)ni * r + ni, nj, nk, r);
    // (double-float products; C itself, with its cancellation, is formed in FP64 above)
    cta_gemm_df_r<4>(ni, nk, nj, -1.0, Mv, Zv, 0.0, Y + ni, r, gsm);                                     // -M Z
    cta_gemm_df_r<4>(nj, nk, nj, 1.0, dense_view(C0, nj, nj, nj), Zv, 0.0, CZ, nk, gsm);                // C Z
    cta_gemm_df_r<4>(nk, nk, nj, 1.0, transpose(Zv), dense_view(CZ, nj, nk, nk), 0.0, pp.ZCZ, nk, gsm);  // Z^T C Z
    if (threadIdx.x == 0) *jb.r = r;
  }
}

// (2) F' = Y^T F Y
__global__ void __launch_bounds__(NT, 2) k_pm_fprime(Tables t, const PJob* __restrict__ jobs,
                                                  const int* __restrict__ order, int n_jobs, double* slots,
                                                  const long long* off, int max_m, double* scratch) {
  __shared__ double sm[GEMM_SMEM_WIDE];
  double* FY = scratch + (size_t)blockIdx.x * pm_cta_doubles(max_m);
  for (int q = blockIdx.x; q < n_jobs; q += gridDim.x) {
    const int jid = order[q];
    const PJob jb = jobs[jid];
    const int i = jb.i, j = jb.j;
    const int ni = t.n_osv[i], nj = (i == j) ? 0 : t.n_osv[j];
    const int m = ni + nj, r = *jb.r, nk = r - ni;
    const PmPair pp = pm_pair(slots, off, jid, m);
    const View Fv = pair_view(t, t.F, i, j, i, j);
    if (i == j) {
      for (int idx = threadIdx.x; idx < m * m; idx += NT) pp.Fp[idx] = Fv.get(idx / m, idx % m);
      __syncthreads();
      continue;
    }
    // F Y: the first ni columns of Y are unit vectors
    for (int idx = threadIdx.x; idx < m * ni; idx += NT)
      FY[(size_t)(idx / ni) * r + idx % ni] = Fv.get(idx / ni, idx % ni);
    cta_gemm_df(m, nk, m, 1.0, Fv, dense_view(pp.Y + ni, m, nk, r), 0.0, FY + ni, r, sm);
    cta_gemm_df(r, r, m, 1.0, transpose(dense_view(pp.Y, m, r, r)), dense_view(FY, m, r, r), 0.0, pp.Fp, r, sm);
  }
}

// (3a) F' symmetrised in FP32, tridiagonalised, Z of the reflectors
template <class T>
__global__ void __launch_bounds__(NT, 3)
    k_pm_eig_a(const PJob* __restrict__ jobs, const int* __restrict__ order, int n_jobs, double* slots,
               const long long* off, const int* mdim, int max_m, double* scratch) {
  extern __shared__ double esm_raw[];   // eigen-solver scratch: 4 max_m + 33 elements
  T* esm = reinterpret_cast<T*>(esm_raw);
  const size_t M2 = (size_t)max_m * max_m;
  T* A = reinterpret_cast<T*>(scratch + (size_t)blockIdx.x * pm_cta_doubles(max_m));
  T* tau = A + M2;
  for (int q = blockIdx.x; q < n_jobs; q += gridDim.x) {
    const int jid = order[q];
    const PJob jb = jobs[jid];
    const int m = mdim[jid], r = *jb.r;
    const PmPair pp = pm_pair(slots, off, jid, m);
    if (pm_eig<T>(pp.wk, m).hdr[3]) continue;
    for (int idx = threadIdx.x; idx < r * r; idx += NT) {
      const int a = idx / r, b = idx % r;
      A[idx] = (T)(0.5 * (pp.Fp[idx] + pp.Fp[(size_t)b * r + a]));
    }
    __syncthreads();
    pm_tridiag(A, r, pm_eig<T>(pp.wk, m), tau, esm);
  }
}

// (3c) eig(F') completed: W, e~
template <class T>
__global__ void __launch_bounds__(NT, 3)
    k_pm_eig_c(const PJob* __restrict__ jobs, const int* __restrict__ order, int n_jobs, double* slots,
               const long long* off, const int* mdim, int max_m, double* scratch, int* err) {
  extern __shared__ double esm_raw[];   // eigen-solver scratch: 4 max_m + 33 elements
  T* esm = reinterpret_cast<T*>(esm_raw);
  const size_t M2 = (size_t)max_m * max_m;
  T* A = reinterpret_cast<T*>(scratch + (size_t)blockIdx.x * pm_cta_doubles(max_m));
  T* ew = A + M2;               // in-CTA solve of a pair whose chase record overflowed
  T* eb = ew + max_m;
  T* tau = eb + max_m;
  for (int q = blockIdx.x; q < n_jobs; q += gridDim.x) {
    const int jid = order[q];
    const PJob jb = jobs[jid];
    const int m = mdim[jid], r = *jb.r;
    const PmPair pp = pm_pair(slots, off, jid, m);
    const PmEig<T> w = pm_eig<T>(pp.wk, m);
    if (w.hdr[3]) continue;
    const T* ev = w.d;
    if (w.hdr[0] == 2) {
      for (int idx = threadIdx.x; idx < r * r; idx += NT) {
        const int a = idx / r, b = idx % r;
        A[idx] = (T)(0.5 * (pp.Fp[idx] + pp.Fp[(size_t)b * r + a]));
      }
      __syncthreads();
      if (cta_syev_cm(A, r, r, ew, w.Z, r, eb, tau, esm) && threadIdx.x == 0) atomicOr(err, ERR_EIG);
      ev = ew;
    } else {
      apply_qr_record_cm(w.Z, r, r, w.swp, w.hdr[1], w.rot);
    }
    for (int idx = threadIdx.x; idx < r * r; idx += NT) {   // W[a][t] = component a of eigenvector t
      const int tv = idx / r, a = idx % r;
      pp.W[(size_t)a * r + tv] = (double)w.Z[idx];
    }
    for (int c = threadIdx.x; c < r; c += NT) {
      pp.et[c] = (double)ev[c];
      if (!isfinite((double)ev[c])) atomicOr(err, ERR_NONFINITE);
    }
    __syncthreads();
  }
}

// (4) X = Y W; S~ = W^T (Y^T S Y) W; F~ = W^T F' W; leftovers.  The products run in
// double-float (~48 bits): W holds FP32 values and Y^T S Y, F' are FP64 with entries
// ~1, so the leftovers (~1e-6) keep ~9 significant digits.  X = Y W (entries up to
// lambda_min(S)^(-1/2)) is double-float as well: U = P X and the leftovers are
// formed from the same X, so its ~2^-48 relative rounding does not move the
// fixed point.
__global__ void __launch_bounds__(NT, 2) k_pm_final(Tables t, const PJob* __restrict__ jobs,
                                                 const int* __restrict__ order, int n_jobs, double* slots,
                                                 const long long* off, int max_m, double* scratch, int* err) {
  __shared__ double sm[GEMM_SMEM_WIDE];
  const size_t M2 = (size_t)max_m * max_m;
  double* T1 = scratch + (size_t)blockIdx.x * pm_cta_doubles(max_m);
  double* St = T1 + M2;
  double* Ft = St + M2;
  const int n = t.n_occ;
  for (int q = blockIdx.x; q < n_jobs; q += gridDim.x) {
    const int jid = order[q];
    const PJob jb = jobs[jid];
    const int i = jb.i, j = jb.j;
    const int ni = t.n_osv[i], nj = (i == j) ? 0 : t.n_osv[j];
    const int m = ni + nj, r = *jb.r, nk = r - ni;
    const PmPair pp = pm_pair(slots, off, jid, m);
    const View Wv = dense_view(pp.W, r, r, r);
    if (i != j) {
      cta_gemm_df(m, r, r, 1.0, dense_view(pp.Y, m, r, r), Wv, 0.0, jb.X, m, sm);       // X = Y W
      if (jb.Sh) {
        for (int idx = threadIdx.x; idx < ni * r; idx += NT) T1[idx] = pp.W[idx];      // (Y^T S Y) W, top rows
        cta_gemm_df(nk, r, nk, 1.0, dense_view(pp.ZCZ, nk, nk, nk), dense_view(pp.W + (size_t)ni * r, nk, r, r), 0.0,
                    T1 + (size_t)ni * r, r, sm);
      }
    } else {
      for (int idx = threadIdx.x; idx < m * r; idx += NT) jb.X[(size_t)(idx / r) * m + idx % r] = pp.W[idx];
      if (jb.Sh) cta_gemm_df(r, r, r, 1.0, dense_view(t.S[t.sf_id[i * n + i]], ni, ni, ni), Wv, 0.0, T1, r, sm);
    }
    for (int c = threadIdx.x; c < r; c += NT) jb.et[c] = pp.et[c];
    if (!jb.Sh) {               // FP64 form: the basis is polished afterwards (solve_oz.cu)
      __syncthreads();
      continue;
    }
    cta_gemm_df(r, r, r, 1.0, transpose(Wv), dense_view(T1, r, r, r), 0.0, St, r, sm);      // S~
    cta_gemm_df(r, r, r, 1.0, dense_view(pp.Fp, r, r, r), Wv, 0.0, T1, r, sm);
    cta_gemm_df(r, r, r, 1.0, transpose(Wv), dense_view(T1, r, r, r), 0.0, Ft, r, sm);      // F~
    const double fh = 0.5 * (t.f_occ[i * n + i] + t.f_occ[j * n + j]);
    for (int idx = threadIdx.x; idx < r * r; idx += NT) {
      const int a = idx / r, b = idx % r;
      const double sh = St[idx] - (a == b ? 1.0 : 0.0);
      const double gh = Ft[idx] - (a == b ? pp.et[a] : 0.0) - fh * sh;
      jb.Sh[idx] = (float)sh;
      jb.Gh[idx] = (float)gh;
      if (!isfinite(sh) || !isfinite(gh)) atomicOr(err, ERR_NONFINITE);
    }
    __syncthreads();
  }
}

size_t precond_mixed_slot_doubles(int m) { return pm_slot_doubles(m); }

size_t precond_mixed_scratch_doubles(int max_m, int n_cta) { return (size_t)n_cta * pm_cta_doubles(max_m); }

constexpr int PM_SMEM = 200 * 1024;

int launch_precond_mixed(const Tables& t, double tau_s, const PJob* jobs, const int* order, int n_jobs, int max_m, int max_n,
                         const int* m_sorted, double* slots, const long long* off, const int* mdim, double* scratch,
                         int n_cta, int num_sms, int* err, cudaStream_t st) {
  if (!n_jobs) return 0;
  const size_t sm_d = ((size_t)4 * max_m + 33) * sizeof(double) + (size_t)max_m * sizeof(int);
  const size_t sm_t = ((size_t)4 * max_m + 33) * sizeof(float);
  const int nsm = max_m < 200 ? max_m : 200;         // 2 nsm 32 doubles: 102 KB at most
  if (sm_d > 160 * 1024) return -1;
  int nmax = max_n, jmax = max_m;
  while (((size_t)nmax * (nmax + 1) + nmax) * sizeof(double) > PM_SMEM) nmax--;
  while (2 * (size_t)jmax * (jmax | 1) * sizeof(float) > PM_SMEM) jmax--;
  const size_t sm_c = ((size_t)nmax * (nmax + 1) + nmax) * sizeof(double);
  for (const void* fn : {(const void*)k_pm_overlap_a, (const void*)k_pm_overlap_c, (const void*)k_pm_chol, (const void*)k_pm_jacobi,
                         (const void*)k_pm_eig_a<float>, (const void*)k_pm_chase<double>, (const void*)k_pm_chase<float>,
                         (const void*)k_pm_eig_c<float>})
    if (allow_dynamic_smem(fn) != cudaSuccess) return -1;
  const int lpw = std::min(32, std::max(1, (n_jobs + 4 * num_sms - 1) / (4 * num_sms)));
  const int n_chase = (n_jobs + lpw - 1) / lpw;
  // Jacobi costs ~2.5 ns per r^3 and SM, the three-step QR a serial ~3 ms and ~1.3 ns: Jacobi below their crossing
  // (32 orbitals, 300 pairs of ~54: 2.7 ms against ~5; 128 orbitals, 1584 pairs of ~92: 23 against 15)
  double r3 = 0.0;
  for (int q = 0; q < n_jobs; q++) r3 += (double)m_sorted[q] * m_sorted[q] * m_sorted[q];
  const bool jacobi = r3 < 2.6e6 * num_sms;
  k_pm_chol<<<n_cta, NT, sm_c, st>>>(t, tau_s, jobs, order, n_jobs, slots, off, max_m, nmax, scratch);
  k_pm_overlap_a<<<n_cta, NT, sm_d, st>>>(t, jobs, order, n_jobs, slots, off, max_m, scratch);
  k_pm_chase<double><<<n_chase, 32, 64 * nsm * 8, st>>>(t, jobs, order, n_jobs, slots, off, mdim, 0, lpw, nsm, err);
  k_pm_overlap_c<<<n_cta, NT, sm_d, st>>>(t, tau_s, jobs, order, n_jobs, slots, off, max_m, scratch, err);
  k_pm_fprime<<<n_cta, NT, 0, st>>>(t, jobs, order, n_jobs, slots, off, max_m, scratch);
  // by size, so that the smaller ones share an SM: up to order 72 five CTAs, up to 104 two (m_sorted descends)
  int j0 = 0;
  for (int cls = 0; cls < 3 && jacobi; cls++) {
    const int cap = cls == 0 ? max_m : (cls == 1 ? 104 : 72), next = cls == 0 ? 104 : (cls == 1 ? 72 : 0);
    int j1 = j0;
    while (j1 < n_jobs && m_sorted[j1] > next) j1++;
    if (j1 == j0) continue;
    const int jm = cap < jmax ? cap : jmax;
    const size_t sm_j = 2 * (size_t)jm * (jm | 1) * sizeof(float);
    k_pm_jacobi<<<j1 - j0 < n_cta ? j1 - j0 : n_cta, NT_J, sm_j, st>>>(jobs, order + j0, j1 - j0, slots, off, mdim, jm, err);
    note_launch(1);
    j0 = j1;
  }
  k_pm_eig_a<float><<<n_cta, NT, sm_t, st>>>(jobs, order, n_jobs, slots, off, mdim, max_m, scratch);
  k_pm_chase<float><<<n_chase, 32, 64 * nsm * 4, st>>>(t, jobs, order, n_jobs, slots, off, mdim, 1, lpw, nsm, err);
  k_pm_eig_c<float><<<n_cta, NT, sm_t, st>>>(jobs, order, n_jobs, slots, off, mdim, max_m, scratch, err);
  k_pm_final<<<n_cta, NT, 0, st>>>(t, jobs, order, n_jobs, slots, off, max_m, scratch, err);
  note_launch(9);
  return 0;
}

}  // namespace osv

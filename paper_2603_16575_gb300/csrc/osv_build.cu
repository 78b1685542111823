// A0: OSV generation.  T_ii from the RI integrals (Eq. mp2_tkk, positive
// denominator e_a + e_b - 2 f_ii), its eigen-decomposition (Eq. osv_gen; FP64, or
// double-float for the mixed form)
// and the selection omega >= l_osv of Algorithm 3, all on the GPU.
#include <algorithm>

#include "eig.cuh"
#include "eig_topk.h"
#include "internal.h"

namespace osv {

// A(a, P) = B[i,a,P] and its transpose, read straight from the source (stored
// or regenerated).
struct BiRows {
  BSrc s;
  int i;
  __device__ __forceinline__ double get(int a, int P) const { return s.get(i, a, P); }
};
struct BiCols {
  BSrc s;
  int i;
  __device__ __forceinline__ double get(int P, int b) const { return s.get(i, b, P); }
};

// One 64x64 tile (tr >= tc) of T_i = (B_i B_i^T) / (e_a + e_b - 2 f_ii); the
// mirror tile is written from the same accumulators.
__global__ void __launch_bounds__(NT) k_tii(BSrc src, const double* __restrict__ e_vir,
                                            const double* __restrict__ f_occ, int n_occ, int i0,
                                            double* __restrict__ T) {
  __shared__ double sm[GEMM_SMEM_DOUBLES];
  const int nv = src.n_vir, nx = src.n_aux;
  const int b = blockIdx.y, i = i0 + b;
  int t = blockIdx.x, tr = 0;
  while ((tr + 1) * (tr + 2) / 2 <= t) tr++;
  const int tc = t - tr * (tr + 1) / 2;
  double acc[4][4];
#pragma unroll
  for (int u = 0; u < 4; u++)
#pragma unroll
    for (int v = 0; v < 4; v++) acc[u][v] = 0.0;
  tile_mma(nv, nv, nx, tr * TM, tc * TN, BiRows{src, i}, BiCols{src, i}, acc, sm);
  const double f2 = 2.0 * f_occ[(size_t)i * n_occ + i];
  double* Ti = T + (size_t)b * nv * nv;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int u = 0; u < 4; u++)
#pragma unroll
    for (int v = 0; v < 4; v++) {
      const int a = tr * TM + ty + 16 * u, c = tc * TN + tx + 16 * v;
      if (a < nv && c < nv) {
        const double val = acc[u][v] / (e_vir[a] + e_vir[c] - f2);
        Ti[(size_t)a * nv + c] = val;
        Ti[(size_t)c * nv + a] = val;
      }
    }
}

void launch_tii(const BSrc& src, const double* e_vir, const double* f_occ, int n_occ, int i0, int nb,
                double* T, cudaStream_t st) {
  const int nt = (src.n_vir + TM - 1) / TM;
  dim3 grid(nt * (nt + 1) / 2, nb);
  k_tii<<<grid, NT, 0, st>>>(src, e_vir, f_occ, n_occ, i0, T);
  note_launch(1);
}

// ---------------------------------------------------------------- eigen
constexpr int ZSMEM_MAX = 160;   // Z kept in shared memory up to this order
// Orders up to this take one CTA per matrix from start to end: below it the fixed costs of the cluster
// tridiagonalisation and of the top-k path (multisection, inverse iteration) are the larger ones.
constexpr int EIG_FULL_MAX = 16;
constexpr int NT_EIG = 1024;     // threads of the full decomposition (rows of Z, and one warp that chases)
constexpr int EB_DF_MAXN = 1536; // double-float back-transformation: the vector in registers up to this order

// Sign eigenvector t (V[t][0..n), eigenvector-major) so that its largest-magnitude
// entry (lowest index on ties) is positive.  One warp per vector.
__device__ inline void sign_vectors(double* V, int n, int k) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int t = warp; t < k; t += NT_EIG / 32) {
    double* x = V + (size_t)t * n;
    double best = -1.0;
    int bi = n - 1;   // in range when no entry compares (NaN)
    for (int r = lane; r < n; r += 32) {
      const double a = fabs(x[r]);
      if (a > best) { best = a; bi = r; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    if (x[bi] < 0.0)
      for (int r = lane; r < n; r += 32) x[r] = -x[r];
  }
  __syncthreads();
}

// The tail of a full decomposition: eigenvalues ww sorted descending, those >= thr (all when thr <= 0) with
// their vectors, at most kmax.  Z(r, column t) at Zs[r * sr + t * sc]; perm: n ints of shared memory.
__device__ void eig_select(const double* ww, int n, int rc, double thr, int kmax, double* V, double* w, int* kout,
                           int* err, const double* Zs, int sr, int sc, int* perm) {
  __shared__ int s_k;
  __syncthreads();
  // rank of each eigenvalue (descending, ties by index; NaN after every number)
  for (int t = threadIdx.x; t < n; t += NT_EIG) {
    const double x = ww[t];
    int at = 0;
    for (int u = 0; u < n; u++) {
      const double y = ww[u];
      const bool yn = isnan(y), xn = isnan(x);
      at += (yn || xn) ? (xn && !yn) || (xn && yn && u < t) : (y > x || (y == x && u < t));
    }
    perm[at] = t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int k = 0;
    if (thr > 0.0) { while (k < n && ww[perm[k]] >= thr) k++; }
    else k = n;
    if (k > kmax) { k = kmax; atomicOr(err, ERR_SIZE); }
    bool bad = rc != 0;
    for (int t = 0; t < n; t++) bad |= !isfinite(ww[t]);
    if (bad) atomicOr(err, rc ? ERR_EIG : ERR_NONFINITE);
    s_k = k;
    *kout = k;
    for (int t = 0; t < k; t++) w[t] = ww[perm[t]];
  }
  __syncthreads();
  const int k = s_k;
  for (int idx = threadIdx.x; idx < n * k; idx += NT_EIG) {
    const int t = idx / n, r = idx % n;
    V[(size_t)t * n + r] = Zs[(size_t)r * sr + (size_t)perm[t] * sc];
  }
  __syncthreads();
  sign_vectors(V, n, k);
}

// Back-transformation of the kept eigenvectors of the top-k path, one warp per
// (orbital, vector) over the whole GPU (the vectors are independent, and
// orbitals keep different numbers of them): x <- H_0 ... H_{n-3} x with the
// reflectors stored contiguously in the rows of A and tau in the scratch, then
// the sign convention of sign_vectors.
constexpr int EB_WARPS = 8;

// The same back-transformation in double-float for the mixed-form build (its
// reflectors are stored as (hi, lo) pairs by k_eig_tri): the vector
// lives in registers, NJ elements per lane (n <= 32 NJ), and every reflector
// costs FP32 instructions only.
template <int NJ>
__global__ void __launch_bounds__(EB_WARPS * 32) k_eig_back_df(const double* T, int n, int kmax, double* V,
                                                              const int* kout, const double* scratch,
                                                              size_t scr_stride) {
  __shared__ dfl s_tau[EB_DF_MAXN];   // tau as pairs: no global load or FP64 work per reflector
  const int b = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.y * EB_WARPS + warp;
  const int kb = kout[b];
  if ((int)blockIdx.y * EB_WARPS >= kb) return;   // CTA-uniform
  const double* tau = scratch + (size_t)b * scr_stride + 2 * n;
  for (int i = threadIdx.x; i < n; i += EB_WARPS * 32) s_tau[i] = df_from(tau[i]);
  __syncthreads();
  if (t >= kb) return;   // warp-uniform
  const dfl* Ad = reinterpret_cast<const dfl*>(T + (size_t)b * n * n);
  double* x = V + (size_t)b * n * kmax + (size_t)t * n;
  dfl xr[NJ];
#pragma unroll
  for (int j = 0; j < NJ; j++) {
    const int r = 32 * j + lane;
    xr[j] = r < n ? df_from(x[r]) : dfl{0.f, 0.f};
  }
  for (int kk = n - 3; kk >= 0; kk--) {
    const dfl tk = s_tau[kk];
    if (tk.h == 0.f) continue;
    const dfl* vr = Ad + (size_t)kk * n;   // v at columns kk+1 .. n-1 of row kk
    const int j0 = (kk + 1) >> 5;          // register blocks below j0 hold no row > kk
    float sh = 0.f, sl = 0.f;
#pragma unroll
    for (int j = 0; j < NJ; j++) {
      if (j < j0) continue;   // warp-uniform
      const int r = 32 * j + lane;
      if (r > kk && r < n) df_acc(sh, sl, vr[r], xr[j]);
    }
    dfl s = df_norm(sh, sl);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = df_add(s, df_shfl_xor(s, o));
    const dfl ns = df_neg(df_mul(s, tk));
#pragma unroll
    for (int j = 0; j < NJ; j++) {
      if (j < j0) continue;
      const int r = 32 * j + lane;
      if (r > kk && r < n) xr[j] = df_fma1(ns, vr[r], xr[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < NJ; j++) {
    const int r = 32 * j + lane;
    if (r < n) x[r] = df_to(xr[j]);
  }
  __syncwarp();
  double best = -1.0;
  int bi = n - 1;   // in range when no entry compares (NaN)
  for (int r = lane; r < n; r += 32) {
    const double a = fabs(x[r]);
    if (a > best) { best = a; bi = r; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
  }
  if (x[bi] < 0.0)
    for (int r = lane; r < n; r += 32) x[r] = -x[r];
}
__global__ void __launch_bounds__(EB_WARPS * 32) k_eig_back(const double* T, int n, int kmax, double* V,
                                                           const int* kout, const double* scratch,
                                                           size_t scr_stride) {
  const int b = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.y * EB_WARPS + warp;
  if (t >= kout[b]) return;   // warp-uniform
  const double* A = T + (size_t)b * n * n;
  const double* tau = scratch + (size_t)b * scr_stride + 2 * n;
  double* x = V + (size_t)b * n * kmax + (size_t)t * n;
  for (int kk = n - 3; kk >= 0; kk--) {
    const double tk = tau[kk];
    if (tk == 0.0) continue;
    const int L = n - kk - 1;
    const double* vr = A + (size_t)kk * n + kk + 1;
    double* xs = x + kk + 1;
    double s = 0.0;
    for (int r = lane; r < L; r += 32) s = fma(vr[r], xs[r], s);
    s = tk * warp_sum(s);
    for (int r = lane; r < L; r += 32) xs[r] = fma(-vr[r], s, xs[r]);
    __syncwarp();
  }
  double best = -1.0;
  int bi = n - 1;   // in range when no entry compares (NaN)
  for (int r = lane; r < n; r += 32) {
    const double a = fabs(x[r]);
    if (a > best) { best = a; bi = r; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
  }
  if (x[bi] < 0.0)
    for (int r = lane; r < n; r += 32) x[r] = -x[r];
}

// Orders up to EIG_FULL_MAX: the whole decomposition by one CTA, everything in shared memory.
__global__ void __launch_bounds__(NT_EIG) k_eig_small(double* T, int n, double thr, int kmax, double* V, double* w,
                                                  int* kout, double* scratch, int* err) {
  extern __shared__ double dyn[];
  const int b = blockIdx.x, ldz = n + 1;
  double* scr = scratch + (size_t)b * eig_osv_scratch_doubles(n, kmax);
  double* ww = scr + 2 * n;
  double* sm = dyn + (size_t)n * ldz;
  const int rc = cta_syev<NT_EIG>(T + (size_t)b * n * n, n, n, ww, dyn, ldz, scr, scr + n, sm);
  eig_select(ww, n, rc, thr, kmax, V + (size_t)b * n * kmax, w + (size_t)b * kmax, kout + b, err, dyn, ldz, 1,
             reinterpret_cast<int*>(sm));
}

// Every eigenpair of a tridiagonalised matrix (k_eig_tri): Z from the reflectors, then the implicit QR, one
// thread chasing and recording rotations into one half of the matrix's storage (free once Z is formed)
// while the other warps apply the previous record to the rows of Z, one thread a row (column-major, so the accesses of
// a warp are contiguous; in shared memory up to ZSMEM_MAX).  Bound by the chase (a chain of ~1.6 n^2
// rotations of ~20 dependent FP64 operations; the application keeps clear of it: with its rows off the
// chase's sub-partition the time is the same).  Against a CTA that waits for each rotation and ~28 operations a
// rotation: 24 matrices of order 120 27 -> 13.1 ms (15.4 with the longer rotation), 10 of order 50 6.5 -> 3.0 (3.6).
__global__ void __launch_bounds__(NT_EIG) k_eig_full(double* T, int n, double thr, int kmax, double* V, double* w,
                                                 int* kout, double* scratch, int* err) {
  extern __shared__ double dyn[];
  const int b = blockIdx.x, tid = threadIdx.x;
  double* A = T + (size_t)b * n * n;
  double* scr = scratch + (size_t)b * eig_osv_scratch_doubles(n, kmax);
  double* dv = dyn;
  double* ev = dyn + n;
  double* Z = n <= ZSMEM_MAX ? dyn + 2 * n : scr + 3 * n;
  __shared__ int s_rc, s_ns[2];
  cta_form_z_cm<NT_EIG, double, true>(A, n, n, scr + 2 * n, Z, n, dv, ev);
  for (int t = tid; t < n; t += NT_EIG) {
    dv[t] = scr[t];
    ev[t] = t + 1 < n ? scr[n + t] : 0.0;
  }
  __syncthreads();
  // two records of at most 32 n rotations each (a sweep is below n): sweeps as int pairs, then (c, s) pairs
  const int half = n * n / 2, cap_s = half / 8, cap_r = min((half - cap_s) / 2, 32 * n);
  const int max_sweeps = 40 * n + 100;        // of all records: a matrix that never deflates (NaN) ends here
  int rc = 2, total = 0;
  if (tid == 0) s_rc = 2;
  for (int c = 0; c <= max_sweeps; c++) {     // each record holds at least one sweep
    double* rec = A + (size_t)(c & 1) * half;
    const double* old = A + (size_t)((c + 1) & 1) * half;
    if (tid == 0) {
      int ns = 0;
      if (rc == 2) s_rc = tridiag_qr_record(dv, ev, n, reinterpret_cast<int*>(rec), cap_s, rec + cap_s, cap_r, &ns, true);
      total += ns;
      if (rc == 2 && s_rc == 2 && total > max_sweeps) s_rc = 1;
      s_ns[c & 1] = ns;
    } else if (tid >= 32 && c > 0) {
      const int* swp = reinterpret_cast<const int*>(old);
      const int ns = s_ns[(c + 1) & 1];
      for (int row = tid - 32; row < n; row += NT_EIG - 32) {
        double* zr = Z + row;
        const double* cs = old + cap_s;
        for (int q = 0; q < ns; q++) {
          const int l = swp[2 * q], h = swp[2 * q + 1];
          double carry = zr[(size_t)l * n];
          for (int k = l; k < h; k++, cs += 2) {
            const double co = cs[0], si = cs[1];
            const double y = zr[(size_t)(k + 1) * n];
            zr[(size_t)k * n] = co * carry + si * y;
            carry = -si * carry + co * y;
          }
          zr[(size_t)h * n] = carry;
        }
      }
    }
    __syncthreads();
    if (rc != 2) break;   // the last record has been applied
    rc = s_rc;
    __syncthreads();
  }
  double* ww = scr + n;   // the sub-diagonal is no longer needed
  for (int t = tid; t < n; t += NT_EIG) ww[t] = dv[t];
  eig_select(ww, n, rc, thr, kmax, V + (size_t)b * n * kmax, w + (size_t)b * kmax, kout + b, err, Z, 1, n,
             reinterpret_cast<int*>(ev));
}

void launch_eig_osv(double* T, int nb, int nv, double thr, int kmax, double* V, double* w, int* k,
                    double* scratch, int* err, bool dfl_tridiag, const int* nclu, cudaStream_t st, cudaStream_t st_qr,
                    cudaEvent_t fork) {
  if (nv <= EIG_FULL_MAX) {
    const size_t smem = ((size_t)nv * (nv + 1) + 4 * nv + 64) * sizeof(double);
    k_eig_small<<<nb, NT_EIG, smem, st>>>(T, nv, thr, kmax, V, w, k, scratch, err);
    note_launch(1);
  } else if (thr > 0.0) {
    const bool df = dfl_tridiag && nv > ZSMEM_MAX;   // FP64 in both forms below
    launch_eig_topk(T, nb, nv, thr, kmax, V, w, k, scratch, err, df, df && nv <= EB_DF_MAXN, nclu, st);
  } else {
    launch_eig_tridiag(T, nb, nv, kmax, scratch, err, nclu, st);
    const size_t smem = (2 * (size_t)nv + (nv <= ZSMEM_MAX ? (size_t)nv * nv : 0)) * sizeof(double);
    allow_dynamic_smem((const void*)k_eig_full);
    if (fork && cudaEventRecord(fork, st) == cudaSuccess && cudaStreamWaitEvent(st_qr, fork, 0) == cudaSuccess) st = st_qr;
    k_eig_full<<<nb, NT_EIG, smem, st>>>(T, nv, thr, kmax, V, w, k, scratch, err);
    note_launch(1);
  }
}

void launch_eig_back(double* T, int nb, int nv, double thr, int kmax, double* V, const int* k, double* scratch,
                     bool dfl_tridiag, cudaStream_t st) {
  if (nv <= EIG_FULL_MAX || !(thr > 0.0)) return;   // the other paths form the eigenvectors themselves
  dim3 grid(nb, (std::min(kmax, nv) + EB_WARPS - 1) / EB_WARPS);
  const size_t ss = eig_osv_scratch_doubles(nv, kmax);
  if (dfl_tridiag && nv > ZSMEM_MAX && nv <= EB_DF_MAXN) {   // reflectors stored as pairs
    if (nv <= 640) k_eig_back_df<20><<<grid, EB_WARPS * 32, 0, st>>>(T, nv, kmax, V, k, scratch, ss);
    else if (nv <= 1280) k_eig_back_df<40><<<grid, EB_WARPS * 32, 0, st>>>(T, nv, kmax, V, k, scratch, ss);
    else k_eig_back_df<48><<<grid, EB_WARPS * 32, 0, st>>>(T, nv, kmax, V, k, scratch, ss);
  } else {
    k_eig_back<<<grid, EB_WARPS * 32, 0, st>>>(T, nv, kmax, V, k, scratch, ss);
  }
  note_launch(1);
}

__global__ void k_pack_q(const double* V, const double* w, int nv, int kmax, const int* k,
                         double* const* Qdst, double* const* wdst) {
  const int b = blockIdx.y;
  const int kb = k[b];
  const double* Vb = V + (size_t)b * nv * kmax;
  double* Q = Qdst[b];
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < nv * kb; idx += gridDim.x * blockDim.x) {
    const int r = idx / kb, t = idx % kb;
    Q[idx] = Vb[(size_t)t * nv + r];
  }
  if (blockIdx.x == 0)
    for (int t = threadIdx.x; t < kb; t += blockDim.x) wdst[b][t] = w[(size_t)b * kmax + t];
}

void launch_pack_q(const double* V, const double* w, int nb, int nv, int kmax, const int* k,
                   double* const* Qdst, double* const* wdst, cudaStream_t st) {
  dim3 grid(32, nb);
  k_pack_q<<<grid, 256, 0, st>>>(V, w, nv, kmax, k, Qdst, wdst);
  note_launch(1);
}

}  // namespace osv

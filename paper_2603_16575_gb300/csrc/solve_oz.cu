// FP64 form, A3-A4 on the tensor cores: every pair's preconditioner basis polished to FP64
// accuracy, and the amplitude iterations of many fragments at once in that basis.
//
// With T_p = X_p Y_p X_p^T (T starts at 0 and every update of Algorithm 7 lies in the span of X_p),
// U_p = P_p X_p orthonormal and F diagonal in it, Eq. (res_close) reads
//   R~_p = K~_p - D_p o Y_p + C_p,   C_p = sum_terms c_t Sigma_pq op(Y_q) Sigma_pq^T,
// K~_p = X_p^T K_p X_p, Sigma_pq = U_p^T U_q, and the update is Y_p <- (K~_p + C_p) / D_p: the
// products of the pair with itself (half of the operations of the raw-basis residual) are gone.
// The rest are two products per coupling term, both FP64 contractions of tc_oz.cuh:
//   W_t^T = Sigma_pq op(Y_q)^T    digits written by the epilogue, one exponent per matrix
//   C_p   = sum_t c_t Sigma_pq W_t
// A sweep is four launches over all fragments: W, C, the element-wise update with the digits of
// the new Y, and the convergence test, whose flags make the next sweep leave finished fragments out.
//
// The exponents are bounds, so no pass over W is needed for its largest element: |W_t| <= the norm
// of op(Y_q), since the rows of Sigma_pq are no longer than 1.  The slices hold 63 bits below the
// bound, ten more than the mantissa.
#include "oz_split.cuh"
#include "pairview.cuh"
#include "row_index.h"

namespace osv {

// ---------------------------------------------------------------- basis polish
// Steps of the refinement of Ogita and Aishima (Japan J. Indust. Appl. Math. 35 (2018) 1007) on the basis
// U0 = P X: with S1 = U0^T U0 and F1 = U0^T e U0 formed from U0 itself (entries of order 1; X^T S X would carry
// eps |X|^2, X reaching lambda_min(S)^(-1/2)) and R = 1 - S1,
//   A = F1 + (R F1 + F1 R) / 2 to first order in R, the Fock matrix of the orthonormalised basis U0 (1 + R / 2);
//   U <- U0 (1 + R / 2) G (1 + E), X likewise (two contractions), e~ = diag(A),
// G the Jacobi rotations of the pairs of levels with |A_ab| > 1e-3 |A_bb - A_aa|, E_ab = A_ab / (A_bb - A_aa) of the
// rotated A for the others.  A step squares the errors, so two or three take the FP32 basis (R and the off-diagonal A ~
// 1e-6) to FP64 rounding, groups of close levels four to eleven.  What it takes for these:
//  * an entry of A is known to 8 eps (|A_aa| + |A_bb|) (rounding) and |R|_F^2 max|A| (the second order in R); entries below
//    are left alone, since E or a rotation of what is not known would scramble equal or close levels in every step
//    (E up to 1e-8 is harmless: 1 + E is orthogonal to E^2);
//  * every pair of close levels is rotated, a list at a time in index order, whatever their number: sums over a list do not
//    depend on timing.  Above POL_MAX pairs (a group of 24 and more) the rotations act on a G kept in IE and E = 0.
// The last step is one that finds nothing left to do: |R| < 1e-9 and every |A_ab| either below 1e-8 of its gap or
// within rounding (16 eps max|A|); *ok says whether this one was, and the caller repeats the step for the others.
constexpr int POL_MAX = 256;      // close pairs listed at a time
constexpr int POL_REC = 1024;     // recorded rotations (lists of up to POL_MAX pairs)
constexpr int POL_SWEEPS = 12;
constexpr double POL_EPS = 2.220446049250313e-16;
__global__ void __launch_bounds__(NT) k_oz_polish(const OzPolish* __restrict__ jobs, int n_jobs, int max_r,
                                                  double* scratch) {
  __shared__ double red[40];
  __shared__ double rcs[2 * POL_REC];                // (c, s) of the recorded rotations
  __shared__ unsigned rec[POL_REC];                  // and their elements of A
  __shared__ unsigned key[POL_MAX], list[POL_MAX];
  __shared__ int s_n, s_rec, wcnt[NT / 32];
  double* A = scratch + (size_t)blockIdx.x * max_r * max_r;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int jq = blockIdx.x; jq < n_jobs; jq += gridDim.x) {
    const OzPolish jb = jobs[jq];
    const int r = jb.r, rr = r * r;
    double* RG = jb.F1;           // R / 2, then R G / 2
    double r2 = 0.0;
    unsigned rm = 0;              // upper word of max|R|
    for (int idx = tid; idx < rr; idx += NT) {
      const int a = idx / r, b = idx % r;
      const double R = (a == b ? 1.0 : 0.0) - 0.5 * (jb.S1[idx] + jb.S1[b * r + a]);
      r2 = fma(R, R, r2);
      rm = max(rm, (unsigned)__double2hiint(R) & 0x7fffffffu);
      A[idx] = 0.5 * (jb.F1[idx] + jb.F1[b * r + a]) + 0.5 * R * (jb.F1[(size_t)a * r + a] + jb.F1[(size_t)b * r + b]);
    }
    if (tid == 0) s_n = s_rec = 0;
    r2 = cta_sum(r2, red);        // ends with a barrier: A is complete
    double em = 0.0;
    for (int a = tid; a < r; a += NT) em = fmax(em, fabs(A[(size_t)a * r + a]));
    em = cta_max(em, red);
    const double second = r2 * em, round_max = 16.0 * POL_EPS * em;
    // |x| of the pair of levels da, db: known to `known`
    auto known = [&](double da, double db) { return fmax(second, 8.0 * POL_EPS * (fabs(da) + fabs(db))); };
    auto close = [&](int idx) {
      const int a = idx / r, b = idx % r;
      if (a >= b) return false;
      const double x = fabs(A[idx]), da = A[(size_t)a * r + a], db = A[(size_t)b * r + b];
      return x > 1e-3 * fabs(db - da) && x > known(da, db);
    };
    bool left = __double2hiint(1e-9) <= (int)rm || !(r2 < 1.0);
    for (int idx = tid; idx < rr; idx += NT) {
      const int a = idx / r, b = idx % r;
      RG[idx] = 0.5 * ((a == b ? 1.0 : 0.0) - 0.5 * (jb.S1[idx] + jb.S1[b * r + a]));
      if (a < b) {
        const double x = fabs(A[idx]), da = A[(size_t)a * r + a], db = A[(size_t)b * r + b];
        if (!(x <= 1e-8 * fabs(db - da))) left |= !(x <= fmax(round_max, known(da, db)));
      }
    }
    left = __syncthreads_or(left);
    if (tid == 0) *jb.ok = !left;
    bool many = false;
    for (int sw = 0; left && sw < POL_SWEEPS; sw++) {
      for (int idx = tid; idx < rr; idx += NT)
        if (close(idx)) {
          const int k = atomicAdd(&s_n, 1);
          if (k < POL_MAX) key[k] = (unsigned)idx;
        }
      __syncthreads();
      const int n = s_n;
      __syncthreads();
      if (tid == 0) s_n = 0;
      if (n == 0) break;
      if (n > POL_MAX && !many) {
        if (sw > 0) break;          // the next step takes them
        many = true;
        for (int idx = tid; idx < rr; idx += NT) jb.IE[idx] = idx / r == idx % r ? 1.0 : 0.0;
        __syncthreads();
      }
      for (int pos = 0; pos < rr;) {
        int cnt = 0;
        if (n <= POL_MAX) {          // all of them, in index order whatever order they were found in
          for (int k = tid; k < n; k += NT) {
            int rank = 0;
            for (int u = 0; u < n; u++) rank += key[u] < key[k];
            list[rank] = key[k];
          }
          cnt = n;
          pos = rr;
        } else {                     // the next POL_MAX in index order
          while (pos < rr && cnt < POL_MAX) {
            const bool f = pos + tid < rr && close(pos + tid);
            const unsigned bal = __ballot_sync(0xffffffffu, f);
            if (lane == 0) wcnt[warp] = __popc(bal);
            __syncthreads();
            int at = cnt + __popc(bal & ((1u << lane) - 1u)), all = cnt;
            for (int w = 0; w < NT / 32; w++) {
              at += w < warp ? wcnt[w] : 0;
              all += wcnt[w];
            }
            if (f && at < POL_MAX) list[at] = (unsigned)(pos + tid);
            __syncthreads();
            pos = all > POL_MAX ? (int)list[POL_MAX - 1] + 1 : pos + NT;
            cnt = min(all, POL_MAX);
          }
        }
        __syncthreads();
        for (int k = 0; k < cnt && (many || s_rec < POL_REC); k++) {
          const int p = list[k] / r, q = list[k] % r;
          const double app = A[(size_t)p * r + p], aqq = A[(size_t)q * r + q], apq = A[(size_t)p * r + q];
          __syncthreads();
          if (!(fabs(apq) > 1e-6 * fabs(aqq - app) && fabs(apq) > known(app, aqq))) continue;   // uniform
          const double th = (aqq - app) / (2.0 * apq);
          const double tt = copysign(1.0, th) / (fabs(th) + sqrt(1.0 + th * th));
          const double c = 1.0 / sqrt(1.0 + tt * tt), s = tt * c;
          for (int u = tid; u < r; u += NT) {
            if (u != p && u != q) {
              const double x = A[(size_t)p * r + u], y = A[(size_t)q * r + u];
              const double nx = c * x - s * y, ny = s * x + c * y;
              A[(size_t)p * r + u] = A[(size_t)u * r + p] = nx;
              A[(size_t)q * r + u] = A[(size_t)u * r + q] = ny;
            }
            const double x = RG[(size_t)u * r + p], y = RG[(size_t)u * r + q];
            RG[(size_t)u * r + p] = c * x - s * y;
            RG[(size_t)u * r + q] = s * x + c * y;
            if (many) {
              const double gx = jb.IE[(size_t)u * r + p], gy = jb.IE[(size_t)u * r + q];
              jb.IE[(size_t)u * r + p] = c * gx - s * gy;
              jb.IE[(size_t)u * r + q] = s * gx + c * gy;
            }
          }
          if (tid == 0) {
            A[(size_t)p * r + p] = app - tt * apq;
            A[(size_t)q * r + q] = aqq + tt * apq;
            A[(size_t)p * r + q] = A[(size_t)q * r + p] = 0.0;
            if (!many) {
              rec[s_rec] = list[k];
              rcs[2 * s_rec] = c;
              rcs[2 * s_rec + 1] = s;
              s_rec++;
            }
          }
          __syncthreads();
        }
      }
      if (!many && s_rec >= POL_REC) break;
    }
    __syncthreads();
    for (int a = tid; a < r; a += NT) jb.et[a] = A[(size_t)a * r + a];
    if (!many) {
      for (int idx = tid; idx < rr; idx += NT) {
        const int a = idx / r, b = idx % r;
        double e = a == b ? 1.0 : 0.0;
        if (a != b) {
          const double da = A[(size_t)a * r + a], db = A[(size_t)b * r + b], gap = db - da, x = fabs(A[idx]), g = fabs(gap);
          if (g > 0.0 && (x <= 1e-8 * g || (left && x <= 1e-3 * g && x > known(da, db)))) e = A[idx] / gap;
        }
        jb.IE[idx] = e;
      }
      __syncthreads();
      for (int k = s_rec - 1; k >= 0; k--) {         // G (1 + E): the rotations on the rows, last one first
        const int p = rec[k] / r, q = rec[k] % r;
        const double c = rcs[2 * k], s = rcs[2 * k + 1];
        for (int u = tid; u < r; u += NT) {
          const double x = jb.IE[(size_t)p * r + u], y = jb.IE[(size_t)q * r + u];
          jb.IE[(size_t)p * r + u] = c * x + s * y;
          jb.IE[(size_t)q * r + u] = c * y - s * x;
        }
        __syncthreads();
      }
    }
    __syncthreads();
    for (int idx = tid; idx < rr; idx += NT) jb.IE[idx] += RG[idx];
    __syncthreads();
  }
}
void launch_oz_polish(const OzPolish* jobs, int n_jobs, int max_r, double* scratch, int n_cta, cudaStream_t st) {
  if (!n_jobs) return;
  k_oz_polish<<<n_cta, NT, 0, st>>>(jobs, n_jobs, max_r, scratch);
  note_launch(1);
}

// ---------------------------------------------------------------- update
// Exponent code of a bound |x| < 2^e.
__device__ __forceinline__ int bound_exp(double x) {
  if (!(x > 0.0)) return oz::EX_ZERO;
  return oz::chunk_exp(oz::exp_field(x));
}

// Digits of row m of op(Y) (r x r; v: 0 Y, 1 Y^T, 2 Y + Y^T) under the exponent code e, one warp.
__device__ __forceinline__ void row_digits(const double* Y, int r, int m, int v, int e, int kpad, uint16_t* dst,
                                           size_t slice, int lane) {
  const bool live = e > oz::EX_ZERO / 2 && e < oz::EX_NAN / 2;
  for (int k = 2 * lane; k < kpad; k += 64) {
    double x[2];
#pragma unroll
    for (int u = 0; u < 2; u++) {
      const int kk = k + u;
      x[u] = 0.0;
      if (kk < r) {
        if (v != 1) x[u] = Y[(size_t)m * r + kk];
        if (v != 0) x[u] += Y[(size_t)kk * r + m];
      }
    }
    long long f0 = live ? oz::fixed63(x[0], (unsigned)(e + 1022)) : 0;
    long long f1 = live ? oz::fixed63(x[1], (unsigned)(e + 1022)) : 0;
#pragma unroll
    for (int s = oz::NSL - 1; s >= 0; s--)
      *reinterpret_cast<uint32_t*>(dst + s * slice + k) = oz::digit_pair(f0, f1, s);
  }
}

// 1 / D of a pair, shared by the fragments that hold it: a division takes ten operations of the FP64 pipe, which issues
// one warp in 64 cycles, and the update is bound by it.
__global__ void __launch_bounds__(NT) k_oz_tables(const OzTable* __restrict__ jobs) {
  const OzTable jb = jobs[blockIdx.x];
  for (int idx = blockIdx.y * NT + threadIdx.x; idx < jb.r * jb.r; idx += gridDim.y * NT)
    jb.iD[idx] = 1.0 / (jb.fij - jb.et[idx / jb.r] - jb.et[idx % jb.r]);
}
// Y, energy and digits of a pair: six FP64 operations an element (maxima by integer compares of the magnitudes),
// four elements a thread in flight.  3400 pairs of order ~56: 0.95 -> 0.35 ms.
constexpr int UPU = 4;
__global__ void __launch_bounds__(NT) k_oz_update(const OzPair* __restrict__ pairs, int n_pairs,
                                                  const int* __restrict__ done, int first, int ld, size_t slice, int nch,
                                                  uint16_t* __restrict__ D, int* __restrict__ ex,
                                                  int* __restrict__ exW, double* __restrict__ pe,
                                                  double* __restrict__ pu) {
  __shared__ double red[40];
  __shared__ unsigned long long rdu[NT / 32];
  __shared__ unsigned ram[NT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = blockIdx.x; q < n_pairs; q += gridDim.x) {
    const OzPair p = pairs[q];
    if (done[p.frag]) continue;
    const int r = p.r, rr = r * r;
    unsigned long long du = 0;       // bits of non-negative doubles order as they do (NaN above all)
    unsigned am = 0;                 // upper word of the largest magnitude
    double ss = 0.0;
    for (int i0 = threadIdx.x; i0 < rr; i0 += UPU * NT) {
      double kt[UPU], id[UPU], c[UPU], yo[UPU];
#pragma unroll
      for (int u = 0; u < UPU; u++) {
        const int idx = min(i0 + u * NT, rr - 1);
        kt[u] = p.Kt[idx];
        id[u] = p.iD[idx];
        c[u] = first ? 0.0 : p.C[idx];
        yo[u] = first ? 0.0 : p.Y[idx];
      }
#pragma unroll
      for (int u = 0; u < UPU; u++) {
        const int idx = i0 + u * NT;
        if (idx >= rr) break;
        const double y = (kt[u] + c[u]) * id[u];
        const unsigned long long d = (unsigned long long)__double_as_longlong(y - yo[u]) & 0x7fffffffffffffffull;
        du = d > du ? d : du;
        am = max(am, (unsigned)__double2hiint(y) & 0x7fffffffu);
        ss = fma(y, y, ss);
        p.Y[idx] = y;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long d = __shfl_xor_sync(0xffffffffu, du, o);
      du = d > du ? d : du;
    }
    am = __reduce_max_sync(0xffffffffu, am);
    if (lane == 0) {
      rdu[warp] = du;
      ram[warp] = am;
    }
    ss = cta_sum(ss, red);       // ends with a barrier: Y, rdu and ram are complete
    for (int u = 0; u < NT / 32; u++) {
      du = rdu[u] > du ? rdu[u] : du;
      am = max(am, ram[u]);
    }
    const bool bad = am >= 0x7ff00000u || (du >> 52) >= 2047;
    double e = 0.0;
    const unsigned mag = row_magic((unsigned)r);
    for (int i0 = threadIdx.x; i0 < rr; i0 += UPU * NT) {
      double kt[UPU], y[UPU], yt[UPU];
#pragma unroll
      for (int u = 0; u < UPU; u++) {
        const int idx = min(i0 + u * NT, rr - 1), a = (int)row_of((unsigned)idx, (unsigned)r, mag);
        kt[u] = p.Kt[idx];
        y[u] = p.Y[idx];
        yt[u] = p.Y[(size_t)(idx - a * r) * r + a];
      }
#pragma unroll
      for (int u = 0; u < UPU; u++)
        if (i0 + u * NT < rr) e = fma(kt[u], fma(2.0, y[u], -yt[u]), e);
    }
    e = cta_sum(e, red);
    if (threadIdx.x == 0) {
      pe[q] = p.diag ? e : 2.0 * e;
      pu[q] = bad ? __longlong_as_double(0x7FF8000000000000ll) : __longlong_as_double((long long)du);
    }
    const int eY = bad ? oz::EX_ZERO : oz::chunk_exp(am >> 20);
    const int eW = bound_exp(bad ? 0.0 : sqrt(ss) * (1.0 + 1e-3));
    for (int v = 0; v < 3; v++) {
      const int id = p.ver[v];
      if (id < 0) continue;
      const int up = (v == 2), ey = eY == oz::EX_ZERO ? eY : eY + up, ew = eW == oz::EX_ZERO ? eW : eW + up;
      if (threadIdx.x < nch) {
        ex[(size_t)id * nch + threadIdx.x] = ey;
        exW[(size_t)id * nch + threadIdx.x] = ew;
      }
      uint16_t* base = D + (size_t)p.vrow[v] * ld;
      for (int m = warp; m < r; m += NT / 32)
        row_digits(p.Y, r, m, v, ey, p.kpad, base + (size_t)m * ld, slice, lane);
    }
    __syncthreads();
  }
}

// One thread per fragment: its energy and largest update from its pairs (in order), the test of
// Algorithm 7, the result record and the flag that stops it.
__global__ void k_oz_converge(const int* __restrict__ pair0, int n_frag, const double* __restrict__ pe,
                              const double* __restrict__ pu, SolveOpts o, double ulps, int it, double* __restrict__ e_prev,
                              int* __restrict__ done, int* __restrict__ left, FragOut* __restrict__ out,
                              const int* __restrict__ out_id) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= n_frag || done[f]) return;
  double e = 0.0, um = 0.0;
  bool nan = false;
  for (int q = pair0[f]; q < pair0[f + 1]; q++) {
    e += pe[q];
    um = fmax(um, pu[q]);
    nan |= isnan(pu[q]);
  }
  int status = ERR_NOCONV;
  if (nan || !isfinite(e) || !isfinite(um)) status = ERR_NONFINITE;
  else if (um < o.tol_update && fabs(e - e_prev[f]) < fmax(o.tol_energy, ulps * fabs(e))) status = 0;
  e_prev[f] = e;
  out[out_id[f]] = FragOut{e, nan ? __longlong_as_double(0x7FF8000000000000ll) : um, it, status};
  if (status != ERR_NOCONV || it == o.max_iter) done[f] = 1;
  else atomicAdd(left, 1);
}

void launch_oz_update(const OzPair* pairs, int n_pairs, const int* done, bool first, int ld, long long rows, int nch, uint16_t* D,
                      int* ex, int* exW, double* pe, double* pu, int n_cta, cudaStream_t st) {
  if (!n_pairs) return;
  k_oz_update<<<n_cta, NT, 0, st>>>(pairs, n_pairs, done, first ? 1 : 0, ld, (size_t)rows * ld, nch, D, ex, exW, pe, pu);
  note_launch(1);
}
void launch_oz_tables(const OzTable* jobs, int n, cudaStream_t st) {
  if (!n) return;
  k_oz_tables<<<dim3(n, 4), NT, 0, st>>>(jobs);
  note_launch(1);
}
void launch_oz_converge(const int* pair0, int n_frag, const double* pe, const double* pu, SolveOpts o, double ulps, int it,
                        double* e_prev, int* done, int* left, FragOut* out, const int* out_id, cudaStream_t st) {
  if (!n_frag) return;
  cudaMemsetAsync(left, 0, sizeof(int), st);
  k_oz_converge<<<(n_frag + 127) / 128, 128, 0, st>>>(pair0, n_frag, pe, pu, o, ulps, it, e_prev, done, left, out, out_id);
  note_launch(1);
}

// T_p = X_p Y_p X_p^T of the listed pairs (the weak pairs and the OSV response use the raw OSV basis); T may
// be Y's own storage.
__global__ void __launch_bounds__(NT) k_oz_raw(const OzPair* __restrict__ pairs, int n_pairs, int max_m,
                                               double* scratch) {
  __shared__ double sm[GEMM_SMEM_WIDE];
  double* W = scratch + (size_t)blockIdx.x * max_m * max_m;
  for (int q = blockIdx.x; q < n_pairs; q += gridDim.x) {
    const OzPair p = pairs[q];
    const View Xv = dense_view(p.X, p.m, p.r, p.m);
    cta_gemm_a(p.m, p.r, p.r, 1.0, Xv, dense_view(p.Y, p.r, p.r, p.r), 0.0, W, p.r, sm);
    cta_gemm_a(p.m, p.m, p.r, 1.0, dense_view(W, p.m, p.r, p.r), transpose(Xv), 0.0, p.T, p.m, sm);
  }
}
void launch_oz_raw(const OzPair* pairs, int n_pairs, int max_m, double* scratch, int n_cta, cudaStream_t st) {
  if (!n_pairs) return;
  k_oz_raw<<<n_cta, NT, 0, st>>>(pairs, n_pairs, max_m, scratch);
  note_launch(1);
}

// ---------------------------------------------------------------- adjoint in the preconditioner basis
// dE/df of a fragment, -sum_j <T~_kj, T_lj> - sum_i <T~_il, T_ik> = -2 sum_j <T~_kj, T_lj> (the second sum is the
// transpose of the first): for k != l the products Sigma_pq op(Y_q) Sigma_pq^T of a coupling, dotted with
// 2 Y_p - Y_p^T by the contraction's epilogue (each of a fragment's nine (k < l, j) once); for k = l the dots of the
// pairs with themselves, formed here.  One CTA per fragment.
__global__ void __launch_bounds__(NT) k_oz_df(const OzDf* __restrict__ frags, int n_frag,
                                              const OzPair* __restrict__ pairs, const double* __restrict__ parts,
                                              double* __restrict__ g) {
  __shared__ double red[40];
  __shared__ double self[6];
  for (int f = blockIdx.x; f < n_frag; f += gridDim.x) {
    const OzDf d = frags[f];
    const int np = d.nc * (d.nc + 1) / 2;
    for (int p = 0; p < np; p++) {
      const OzPair pr = pairs[d.pair0 + p];
      double s = 0.0;
      for (int idx = threadIdx.x; idx < pr.r * pr.r; idx += NT)
        s += (2.0 * pr.Y[idx] - pr.Y[(size_t)(idx % pr.r) * pr.r + idx / pr.r]) * pr.Y[idx];
      s = cta_sum(s, red);
      if (threadIdx.x == 0) self[p] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double* out = g + (size_t)d.out * 9;
      int t = 0;   // dots in the order (k < l), j
      for (int k = 0; k < d.nc; k++)
        for (int l = k; l < d.nc; l++) {
          double s = 0.0;
          for (int j = 0; j < d.nc; j++) {
            if (k == l) {
              const int a = min(k, j), b = max(k, j);
              s += self[a * d.nc - a * (a - 1) / 2 + (b - a)];
            } else {
              for (int q = d.tile0[t]; q < d.tile0[t + 1]; q++)
                for (int u = 0; u < 16; u++) s += parts[(size_t)16 * q + u];
              t++;
            }
          }
          out[k * 3 + l] = out[l * 3 + k] = -2.0 * d.weight * s;
        }
    }
    __syncthreads();
  }
}
void launch_oz_df(const OzDf* frags, int n_frag, const OzPair* pairs, const double* parts, double* g, int n_cta,
                  cudaStream_t st) {
  if (!n_frag) return;
  k_oz_df<<<n_cta, NT, 0, st>>>(frags, n_frag, pairs, parts, g);
  note_launch(1);
}

// W_p = sum_C c_C (2 Y - Y^T) over the contributions of each pair.
__global__ void __launch_bounds__(NT) k_oz_gsum(const OzGradPair* __restrict__ jobs, const GradContrib* __restrict__ con) {
  const OzGradPair jb = jobs[blockIdx.x];
  const int r = jb.r;
  for (int idx = blockIdx.y * NT + threadIdx.x; idx < r * r; idx += gridDim.y * NT) {
    const int tr = (idx % r) * r + idx / r;
    double s = 0.0;
    for (int q = jb.c0; q < jb.c1; q++) s += con[q].weight * (2.0 * con[q].T[idx] - con[q].T[tr]);
    jb.Wy[idx] = s;
  }
}
void launch_oz_gsum(const OzGradPair* jobs, int n_jobs, const GradContrib* con, cudaStream_t st) {
  if (!n_jobs) return;
  k_oz_gsum<<<dim3(n_jobs, 8), NT, 0, st>>>(jobs, con);
  note_launch(1);
}
// W = X W_y X^T and H = X H_y X^T.
__global__ void __launch_bounds__(NT) k_oz_graw(const OzGradPair* __restrict__ jobs, int n_jobs, int max_m,
                                                double* scratch) {
  __shared__ double sm[GEMM_SMEM_WIDE];
  double* A = scratch + (size_t)blockIdx.x * max_m * max_m;
  for (int q = blockIdx.x; q < 2 * n_jobs; q += gridDim.x) {
    const OzGradPair p = jobs[q >> 1];
    const View Xv = dense_view(p.X, p.m, p.r, p.m);
    cta_gemm_a(p.m, p.r, p.r, 1.0, Xv, dense_view((q & 1) ? p.Hy : p.Wy, p.r, p.r, p.r), 0.0, A, p.r, sm);
    cta_gemm_a(p.m, p.m, p.r, 1.0, dense_view(A, p.m, p.r, p.r), transpose(Xv), 0.0, (q & 1) ? p.H : p.W, p.m, sm);
  }
}
void launch_oz_graw(const OzGradPair* jobs, int n_jobs, int max_m, double* scratch, int n_cta, cudaStream_t st) {
  if (!n_jobs) return;
  k_oz_graw<<<n_cta, NT, 0, st>>>(jobs, n_jobs, max_m, scratch);
  note_launch(1);
}

}  // namespace osv

// Occupied-orbital localization (Section 3.2, Algorithm 2): Pipek-Mezey with
// Loewdin charges by Jacobi sweeps.
//   P^A_ij = sum_{alpha in A} C~_alpha,i C~_alpha,j
//   per pair i < j in order: a_ij = sum_A (P^A_ij)^2 - (P^A_ii - P^A_jj)^2 / 4,
//   b_ij = sum_A P^A_ij (P^A_ii - P^A_jj), theta = atan2(b, -a) / 4 (Eq. loc_theta,
//   the branch that maximises L), skipped when |sin theta| < 1e-10; otherwise
//   dL += sqrt(a^2 + b^2)(1 - cos 4 theta) and columns i, j of U and both MO
//   indices of every P^A are rotated.  Sweeps until dL <= l_loc.
// The pairs are sequential (each rotation uses the previous one's P); every
// rotation is spread over the CTA's threads by (k, atom), as in the paper.
// Layout: P [n][n][n_atom] (atom index innermost), U [n][n] row-major.
#include "internal.h"

namespace osv {

constexpr int NT_LOC = 1024;

__global__ void k_pm_charges(const double* __restrict__ C, int n_ao, int n, const int* __restrict__ atom_ao,
                             int n_atom, double* __restrict__ P) {
  const long long tot = (long long)n * n * n_atom;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
    const int A = (int)(e % n_atom);
    const long long ij = e / n_atom;
    const int i = (int)(ij / n), j = (int)(ij % n);
    double s = 0.0;
    for (int al = atom_ao[A]; al < atom_ao[A + 1]; al++) s = fma(C[(size_t)al * n + i], C[(size_t)al * n + j], s);
    P[e] = s;
  }
}

// Deterministic CTA sum over NT_LOC threads (shuffle tree, then the warps in order).
__device__ double loc_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = warp_sum(v);
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < NT_LOC / 32; k++) s += red[k];
    red[32] = s;
  }
  __syncthreads();
  const double r = red[32];
  __syncthreads();
  return r;
}

// out[0] = L, out[1] = dL of the last sweep; status[0] = sweeps, status[1] = 1 if converged.
__global__ void __launch_bounds__(NT_LOC) k_pm_sweeps(double* __restrict__ P, double* __restrict__ U, int n, int n_atom,
                                                      double l_loc, int max_sweeps, double* out, int* status) {
  __shared__ double red[33];
  __shared__ double s_c, s_s;
  __shared__ int s_skip;
  const int tid = threadIdx.x;
  for (int k = tid; k < n * n; k += NT_LOC) U[k] = (k / n == k % n) ? 1.0 : 0.0;
  __syncthreads();
  double dL = 0.0;   // meaningful on thread 0
  int sweeps = 0, conv = 0;
  while (sweeps < max_sweeps) {
    sweeps++;
    dL = 0.0;
    for (int i = 0; i < n; i++)
      for (int j = i + 1; j < n; j++) {
        double pa = 0.0, pb = 0.0;
        const double* Pij = P + ((size_t)i * n + j) * n_atom;
        const double* Pii = P + ((size_t)i * n + i) * n_atom;
        const double* Pjj = P + ((size_t)j * n + j) * n_atom;
        for (int A = tid; A < n_atom; A += NT_LOC) {
          const double x = Pij[A], d = Pii[A] - Pjj[A];
          pa += x * x - 0.25 * d * d;
          pb += x * d;
        }
        const double a = loc_sum(pa, red);
        const double b = loc_sum(pb, red);
        if (tid == 0) {
          const double th = 0.25 * atan2(b, -a);
          double sn, cs;
          sincos(th, &sn, &cs);
          s_skip = fabs(sn) < 1e-10;
          s_c = cs;
          s_s = sn;
          if (!s_skip) dL += sqrt(a * a + b * b) * (1.0 - cos(4.0 * th));
        }
        __syncthreads();
        if (s_skip) continue;
        const double c = s_c, s = s_s;
        for (int k = tid; k < n; k += NT_LOC) {
          const double ui = U[(size_t)k * n + i], uj = U[(size_t)k * n + j];
          U[(size_t)k * n + i] = c * ui + s * uj;
          U[(size_t)k * n + j] = c * uj - s * ui;
        }
        // rows i, j against every other k (the first index), mirrored into the columns
        for (long long e = tid; e < (long long)n * n_atom; e += NT_LOC) {
          const int k = (int)(e / n_atom), A = (int)(e % n_atom);
          if (k == i || k == j) continue;
          double* pik = P + ((size_t)i * n + k) * n_atom + A;
          double* pjk = P + ((size_t)j * n + k) * n_atom + A;
          const double x = *pik, y = *pjk;
          const double nx = c * x + s * y, ny = c * y - s * x;
          *pik = nx;
          *pjk = ny;
          P[((size_t)k * n + i) * n_atom + A] = nx;
          P[((size_t)k * n + j) * n_atom + A] = ny;
        }
        // the (i, j) block: first index, then second index
        for (int A = tid; A < n_atom; A += NT_LOC) {
          double* qii = P + ((size_t)i * n + i) * n_atom + A;
          double* qij = P + ((size_t)i * n + j) * n_atom + A;
          double* qji = P + ((size_t)j * n + i) * n_atom + A;
          double* qjj = P + ((size_t)j * n + j) * n_atom + A;
          const double ri0 = c * *qii + s * *qji, ri1 = c * *qij + s * *qjj;   // row i after the first rotation
          const double rj0 = c * *qji - s * *qii, rj1 = c * *qjj - s * *qij;   // row j
          *qii = c * ri0 + s * ri1;
          *qij = c * ri1 - s * ri0;
          *qji = c * rj0 + s * rj1;
          *qjj = c * rj1 - s * rj0;
        }
        __syncthreads();
      }
    __shared__ int s_done;
    if (tid == 0) s_done = !(dL > l_loc);
    __syncthreads();
    if (s_done) {
      conv = 1;
      break;
    }
  }
  double lsum = 0.0;
  for (long long e = tid; e < (long long)n * n_atom; e += NT_LOC) {
    const int i = (int)(e / n_atom), A = (int)(e % n_atom);
    const double d = P[((size_t)i * n + i) * n_atom + A];
    lsum += d * d;
  }
  const double L = loc_sum(lsum, red);
  if (tid == 0) {
    out[0] = L;
    out[1] = dL;
    status[0] = sweeps;
    status[1] = conv;
  }
}

// ---------------------------------------------------------------- whole-GPU form
// The same sweeps with the atoms spread over a cooperative grid: CTA c owns the
// charge matrices of atoms [c apc, (c+1) apc) (atom-major, upper triangle used,
// odd row stride ld, in shared memory when they fit).
//
// Order.  Rotations that share no orbital commute, so the lexicographic sequence
// (0,1), (0,2), ... of a sweep is run as the 2n - 3 steps t = i + j = 1 .. 2n - 3:
// of two pairs that share an orbital the lexicographically earlier one has the
// smaller t (a larger second index, or a larger first one, raises i + j), so every
// rotation still sees exactly the rotations that precede it in the sequence.  A
// step holds up to n/2 disjoint pairs (i, t - i), which share one grid barrier.
//
// Per step every CTA writes its partial (a, b) of the step's pairs, one grid
// barrier, and every CTA adds the G partials of every pair in the same fixed order,
// so all CTAs take the same angles, skip decisions and dL; each then rotates its
// own atoms and its own rows of U.  A single sequence of n(n-1)/2 barriers bounded
// the former one-rotation-per-barrier form (10 us a rotation: 331 ms for 128
// orbitals, 4 sweeps); here the barrier and the partial sums take about half of a
// step and the FP64 pipe (16 operations per 2 x 2 block of the symmetric matrices,
// P <- R^T P R) the rest: 24 ms for the same case.
//
// The barrier is a counter that only grows, with a bounded wait: a CTA that waits
// too long sets ERR_TIMEOUT and leaves, and the others then time out at their next
// barrier.
constexpr int NT_G = 512;
constexpr long long PM_WAIT_LIMIT = 1ll << 22;   // polls (with a short sleep) before giving up

__device__ bool pm_grid_sync(unsigned* bar, unsigned nblocks, unsigned& target) {
  __shared__ int s_ok;
  target += nblocks;
  if (nblocks == 1) {
    __syncthreads();
    return true;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    volatile unsigned* cnt = bar;
    long long it = 0;
    while ((int)(*cnt - target) < 0 && it < PM_WAIT_LIMIT) {
      __nanosleep(20);
      it++;
    }
    s_ok = (int)(*cnt - target) >= 0;
    __threadfence();
  }
  __syncthreads();
  return s_ok != 0;
}

__global__ void k_pm_charges_am(const double* __restrict__ C, int n, int ld, const int* __restrict__ atom_ao, int n_atom,
                                double* __restrict__ P) {
  const long long tot = (long long)n_atom * n * n;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
    const int A = (int)(e / ((long long)n * n));
    const int ij = (int)(e % ((long long)n * n)), i = ij / n, j = ij % n;
    double s = 0.0;
    for (int al = atom_ao[A]; al < atom_ao[A + 1]; al++) s = fma(C[(size_t)al * n + i], C[(size_t)al * n + j], s);
    P[(size_t)A * n * ld + (size_t)i * ld + j] = s;
  }
}

__device__ double pm_block_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = warp_sum(v);
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < NT_G / 32; k++) s += red[k];
    red[32] = s;
  }
  __syncthreads();
  const double r = red[32];
  __syncthreads();
  return r;
}

// cos and sin of theta = atan2(b, -a) / 4 and the gain sqrt(a^2 + b^2) (1 - cos 4 theta)
// by half-angle formulas (|4 theta| <= pi, so cos 2 theta >= 0 and cos theta > 0), each
// half angle from the sum that does not cancel; b = 0 and values whose squares leave the
// FP64 range take the functions themselves.
__device__ __forceinline__ void pm_angle(double a, double b, double& cs, double& sn, double& gain) {
  const double h2 = a * a + b * b;
  if (b == 0.0 || !(h2 > 1e-280 && h2 < 1e280)) {
    const double th = 0.25 * atan2(b, -a);
    sincos(th, &sn, &cs);
    gain = sqrt(h2) * (1.0 - cos(4.0 * th));
    return;
  }
  const double h = sqrt(h2), c4 = -a / h, s4 = b / h;
  double c2, s2;
  if (c4 >= 0.0) {
    c2 = sqrt(0.5 * (1.0 + c4));
    s2 = 0.5 * s4 / c2;
  } else {
    s2 = copysign(sqrt(0.5 * (1.0 - c4)), s4);
    c2 = 0.5 * s4 / s2;
  }
  cs = sqrt(0.5 * (1.0 + c2));
  sn = 0.5 * s2 / cs;
  gain = a < 0.0 ? b * b / (h - a) : h + a;
}

// Dynamic shared memory: the CTA's matrices (SMEM), then [n/2 + 1] pairs' c and s.
template <bool SMEM>
__global__ void __launch_bounds__(NT_G) k_pm_grid(double* __restrict__ Pg, double* __restrict__ U, int n, int ld,
                                                  int n_atom, int apc, double l_loc, int max_sweeps,
                                                  double2* __restrict__ part, unsigned* bar, double* out, int* status,
                                                  int* err) {
  extern __shared__ double dyn[];
  __shared__ double red[33];
  const int cb = blockIdx.x, G = gridDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int A0 = cb * apc, na = max(0, min(n_atom, A0 + apc) - A0);
  const size_t NN = (size_t)n * ld;
  const int maxp = n / 2 + 1;
  double* P = SMEM ? dyn : Pg + (size_t)A0 * NN;
  double* s_c = dyn + (SMEM ? (size_t)apc * NN : 0);
  double* s_s = s_c + maxp;
  if (SMEM)
    for (size_t e = tid; e < (size_t)na * NN; e += NT_G) dyn[e] = Pg[(size_t)A0 * NN + e];
  for (int k = cb; k < n; k += G)
    for (int q = tid; q < n; q += NT_G) U[(size_t)k * n + q] = (k == q) ? 1.0 : 0.0;
  __syncthreads();
  double dL = 0.0;
  unsigned target = 0;
  int sweeps = 0, conv = 0, buf = 0;
  while (sweeps < max_sweeps) {
    sweeps++;
    double gain_sum = 0.0;
    for (int t = 1; t <= 2 * n - 3; t++, buf ^= 1) {
      const int i0 = max(0, t - n + 1), np = (t - 1) / 2 - i0 + 1;   // pairs (i0 + q, t - i0 - q)
      double2* pp = part + (size_t)buf * maxp * G;
      for (int q = tid; q < np; q += NT_G) {
        const int i = i0 + q, j = t - i;
        double pa = 0.0, pb = 0.0;
        for (int u = 0; u < na; u++) {
          const double* Pa = P + (size_t)u * NN;
          const double x = Pa[(size_t)i * ld + j], d = Pa[(size_t)i * ld + i] - Pa[(size_t)j * ld + j];
          pa += x * x - 0.25 * d * d;
          pb += x * d;
        }
        pp[(size_t)q * G + cb] = make_double2(pa, pb);
      }
      if (!pm_grid_sync(bar, (unsigned)G, target)) {
        if (tid == 0) atomicOr(err, ERR_TIMEOUT);
        return;
      }
      for (int q = warp; q < np; q += NT_G / 32) {
        double a = 0.0, b = 0.0;
        for (int g = lane; g < G; g += 32) {
          const double2 v = __ldcg(pp + (size_t)q * G + g);
          a += v.x;
          b += v.y;
        }
        a = warp_sum(a);
        b = warp_sum(b);
        if (lane == 0) {
          s_c[q] = a;
          s_s[q] = b;
        }
      }
      __syncthreads();
      for (int q = tid; q < np; q += NT_G) {
        double cs, sn, gain;
        pm_angle(s_c[q], s_s[q], cs, sn, gain);
        const bool skip = fabs(sn) < 1e-10;
        s_c[q] = skip ? 1.0 : cs;
        s_s[q] = skip ? 0.0 : sn;
        if (!skip) gain_sum += gain;
      }
      __syncthreads();
      for (int k = cb; k < n; k += G)
        for (int q = tid; q < np; q += NT_G) {
          double* u = U + (size_t)k * n;
          const int i = i0 + q, j = t - i;
          const double ui = u[i], uj = u[j], c = s_c[q], s = s_s[q];
          u[i] = c * ui + s * uj;
          u[j] = c * uj - s * ui;
        }
      // P <- R^T P R.  Orbital groups: the np pairs, then the orbitals that this step
      // leaves alone (below i0, the middle one when t is even, above t - i0).
      const int jmax = t - i0, nlow = i0, nmid = (t & 1) ? 0 : 1, nhigh = n - 1 - jmax;
      const int ng = np + nlow + nmid + nhigh;
      for (int w = warp; w < na * np; w += NT_G / 32) {
        const int p = w % np;
        double* Pa = P + (size_t)(w / np) * NN;
        const int i = i0 + p, j = t - i;
        const double c = s_c[p], s = s_s[p];
        for (int q = p + lane; q < ng; q += 32) {
          if (q == p) {
            double* ii = Pa + (size_t)i * ld + i;
            double* ij = Pa + (size_t)i * ld + j;
            double* jj = Pa + (size_t)j * ld + j;
            const double vii = *ii, vij = *ij, vjj = *jj;
            const double ri0 = c * vii + s * vij, ri1 = c * vij + s * vjj;
            const double rj0 = c * vij - s * vii, rj1 = c * vjj - s * vij;
            *ii = c * ri0 + s * ri1;
            *ij = c * ri1 - s * ri0;
            *jj = c * rj1 - s * rj0;
          } else if (q < np) {          // nested pairs: i < i2 < j2 < j
            const int i2 = i0 + q, j2 = t - i2;
            const double c2 = s_c[q], s2 = s_s[q];
            double* e00 = Pa + (size_t)i * ld + i2;
            double* e01 = Pa + (size_t)i * ld + j2;
            double* e10 = Pa + (size_t)i2 * ld + j;
            double* e11 = Pa + (size_t)j2 * ld + j;
            const double v00 = *e00, v01 = *e01, v10 = *e10, v11 = *e11;
            const double x0 = c * v00 + s * v10, x1 = c * v01 + s * v11;
            const double y0 = c * v10 - s * v00, y1 = c * v11 - s * v01;
            *e00 = c2 * x0 + s2 * x1;
            *e01 = c2 * x1 - s2 * x0;
            *e10 = c2 * y0 + s2 * y1;
            *e11 = c2 * y1 - s2 * y0;
          } else {
            const int r = q - np;
            const int k = r < nlow ? r : (r < nlow + nmid ? t / 2 : jmax + 1 + (r - nlow - nmid));
            double* e0 = Pa + (size_t)min(i, k) * ld + max(i, k);
            double* e1 = Pa + (size_t)min(j, k) * ld + max(j, k);
            const double v0 = *e0, v1 = *e1;
            *e0 = c * v0 + s * v1;
            *e1 = c * v1 - s * v0;
          }
        }
      }
      __syncthreads();
    }
    dL = pm_block_sum(gain_sum, red);   // the same value in every CTA
    if (!(dL > l_loc)) {
      conv = 1;
      break;
    }
  }
  // L = sum_{A, i} (P^A_ii)^2
  double ls = 0.0;
  for (int e = tid; e < na * n; e += NT_G) {
    const double d = P[(size_t)(e / n) * NN + (size_t)(e % n) * (ld + 1)];
    ls += d * d;
  }
  ls = pm_block_sum(ls, red);
  double2* pl = part + (size_t)buf * maxp * G;
  if (tid == 0) pl[cb] = make_double2(ls, 0.0);
  if (!pm_grid_sync(bar, (unsigned)G, target)) {
    if (tid == 0) atomicOr(err, ERR_TIMEOUT);
    return;
  }
  if (cb == 0 && tid < 32) {
    double L = 0.0;
    for (int g = lane; g < G; g += 32) L += __ldcg(&pl[g].x);
    L = warp_sum(L);
    if (tid == 0) {
      out[0] = L;
      out[1] = dL;
      status[0] = sweeps;
      status[1] = conv;
    }
  }
}

// Cooperative whole-GPU launch when every CTA can be resident; returns false if not
// possible (the caller then uses the one-CTA form).
bool launch_pm_localize_grid(const double* C, int n, const int* atom_ao, int n_atom, double l_loc, int max_sweeps,
                             double* P, double* U, double* out, int* status, double* part, unsigned* bar, int* err,
                             int num_sms, cudaStream_t st) {
  int ld = n | 1;   // odd: walking a column of a matrix in shared memory meets every bank
  const size_t nn = (size_t)n * ld;
  int G = std::min(n_atom, num_sms);
  int apc = (n_atom + G - 1) / G;
  G = (n_atom + apc - 1) / apc;
  const size_t ang = 2 * (size_t)(n / 2 + 1) * sizeof(double), smem = (size_t)apc * nn * sizeof(double) + ang;
  const bool use_smem = smem <= 200 * 1024;
  void* fn = use_smem ? (void*)k_pm_grid<true> : (void*)k_pm_grid<false>;
  const size_t dsm = use_smem ? smem : ang;
  if (allow_dynamic_smem(fn) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, NT_G, dsm) != cudaSuccess || per_sm < 1 ||
      per_sm * num_sms < G) {
    cudaGetLastError();
    return false;
  }
  const long long tot = (long long)n_atom * n * n;
  k_pm_charges_am<<<(int)std::min<long long>((tot + 255) / 256, 8LL * num_sms), 256, 0, st>>>(C, n, ld, atom_ao, n_atom, P);
  cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), st);
  double2* part2 = reinterpret_cast<double2*>(part);
  void* args[] = {&P, &U, const_cast<int*>(&n), &ld, const_cast<int*>(&n_atom), &apc, &l_loc, &max_sweeps, &part2, &bar,
                  &out, &status, &err};
  if (cudaLaunchCooperativeKernel(fn, dim3(G), dim3(NT_G), args, dsm, st) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  note_launch(2);
  return true;
}

void launch_pm_localize(const double* C, int n_ao, int n, const int* atom_ao, int n_atom, double l_loc, int max_sweeps,
                        double* P, double* U, double* out, int* status, int num_sms, cudaStream_t st) {
  const long long tot = (long long)n * n * n_atom;
  const int grid = (int)std::min<long long>((tot + 255) / 256, 8LL * num_sms);
  k_pm_charges<<<grid, 256, 0, st>>>(C, n_ao, n, atom_ao, n_atom, P);
  k_pm_sweeps<<<1, NT_LOC, 0, st>>>(P, U, n, n_atom, l_loc, max_sweeps, out, status);
  note_launch(2);
}

}  // namespace osv

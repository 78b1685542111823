// Mixed form, A4 for many fragments at once: the amplitude iterations of solve_mixed.cu (same equations, same
// data: Sigma_pq in FP32, leftovers Sh and Gh of the preconditioner basis in FP32, K~, 1/D and Y as
// double-float pairs) with the coupling products on the tensor cores and a sweep as five launches over all fragments:
//   W_t^T = Sigma_pq op(Y_q)^T, C_p = sum_t c_t Sigma_pq W_t       sliced contractions (tc_oz.cuh, four slices)
//   P_p(Y_p) where a fragment's amplitudes have drifted            FP32 CTA products, a pair per CTA
//   Y_p <- (K~_p + C_p + P_p) / D_p, energies, digits of Y         a pair per CTA
//   convergence and drift                                          a thread per fragment
// Four slices hold 31 bits below an operand's exponent (an FP32 element holds 24): 1 for Sigma (|Sigma| <= 1), one per
// matrix for Y (its largest element), and one per pair for the W of its terms, coefficients included (the largest
// norm of Y times c), so that C_p adds up over all terms in tensor memory and is read once.
//
// One CTA per fragment walked its products one after another, each too small for a CTA (orders 30 to 110): 7 to 19 of
// ~70 TFLOP/s FP32.  Measured, amplitude iterations of all fragments, CTA per fragment -> here: 128 orbitals (2215
// three-orbital fragments, pair orders to 150) 88 -> 58 ms, screened list of 64 orbitals 50.5 -> 44, chain of 100
// 20.0 -> 13.2, 32 orbitals 4.3 -> 4.0.  A sweep at 128 orbitals: W 3.2, C 2.6, update 2.9 ms, leftovers 11 (once).
#include "oz_split.cuh"
#include <algorithm>

#include "pairview.cuh"
#include "row_index.h"

namespace osv {
namespace {

constexpr int NS = oz::MXSOLVE;
constexpr int T = 7 + 8 * (NS - 1);        // fixed-point bits below the exponent: |x| < 2^e -> |F| < 2^T = 2^31

__device__ __forceinline__ float pow2f(int x) { return __int_as_float((x + 127) << 23); }   // -126 <= x <= 127

// Exponent code of a bound |x| < 2^e: rows below 2^-90 count as zero.
__device__ __forceinline__ int exp_code(float m) {
  const int f = (__float_as_int(m) >> 23) & 255;
  return f == 255 ? oz::EX_NAN : (f < 37 ? oz::EX_ZERO : f - 126);
}
__device__ __forceinline__ bool live_code(int e) { return e > oz::EX_ZERO / 2 && e < oz::EX_NAN / 2; }

// Digits of one row by a warp: get(k) for k < K as pairs, zeros up to kpad, under the exponent code e.
template <class Get>
__device__ __forceinline__ void row_digits(const Get& get, int K, int k0, int kpad, int e, uint16_t* dst, size_t slice) {
  const int lane = threadIdx.x & 31;
  const bool live = live_code(e);
  const float s0 = live ? pow2f((T - e) >> 1) : 0.f, s1 = live ? pow2f((T - e) - ((T - e) >> 1)) : 0.f;   // T - e in [-97, 121]
  for (int k = k0 + 2 * lane; k < kpad; k += 64) {
    int f[2];
#pragma unroll
    for (int u = 0; u < 2; u++) {
      const dfl x = k + u < K && live ? get(k + u) : dfl{0.f, 0.f};
      const float a = x.h * s0 * s1;       // exact, below 2^31
      const int ia = __float2int_rn(a);
      f[u] = ia + __float2int_rn((a - (float)ia) + x.l * s0 * s1);
    }
#pragma unroll
    for (int s = NS - 1; s >= 0; s--) *reinterpret_cast<uint32_t*>(dst + s * slice + k) = oz::digit_pair32(f[0], f[1], s);
  }
}

// ---------------------------------------------------------------- Sigma
// Digits of an overlap Sigma (lo x hi, FP32) in both orientations under the exponent 1; one CTA per pair couple,
// through shared memory (cap floats) when it fits.
__global__ void __launch_bounds__(NT) k_mx_sigma(const MxSigma* __restrict__ jobs, int n_jobs, int ld, size_t slice, int cap,
                                                 uint16_t* __restrict__ D) {
  extern __shared__ float ssm[];
  const int warp = threadIdx.x >> 5;
  for (int q = blockIdx.x; q < n_jobs; q += gridDim.x) {
    const MxSigma jb = jobs[q];
    const int rl = jb.rl, rh = jb.rh, pitch = rh | 1;
    const bool in = rl * pitch <= cap;
    if (in) {
      for (int idx = threadIdx.x; idx < rl * rh; idx += NT) ssm[(idx / rh) * pitch + idx % rh] = jb.S[idx];
      __syncthreads();
    }
    const float* S = in ? ssm : jb.S;
    const int ls = in ? pitch : rh;
    for (int w = warp; w < rl + rh; w += NT / 32) {
      const bool row = w < rl;
      const int r = row ? w : w - rl, K = row ? rh : rl, kpad = (K + oz::BK - 1) / oz::BK * oz::BK;
      const float* p = row ? S + (size_t)r * ls : S + r;
      const size_t st = row ? 1 : ls;
      row_digits([&](int k) { return dfl{p[k * st], 0.f}; }, K, 0, kpad, 1,
                 D + ((size_t)(row ? jb.lo.row : jb.hi.row) + r) * ld, slice);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- pair tables
// K~ and 1 / D of a pair as double-float pairs (shared by the fragments that hold the pair).
__global__ void __launch_bounds__(NT) k_mx_tables(const MxTable* __restrict__ jobs) {
  const MxTable jb = jobs[blockIdx.x];
  const int r = jb.r;
  for (int idx = blockIdx.y * NT + threadIdx.x; idx < r * r; idx += gridDim.y * NT) {
    jb.Kd[idx] = df_from(jb.Kt[idx]);
    jb.iD[idx] = df_from(1.0 / (jb.fij - jb.et[idx / r] - jb.et[idx % r]));
  }
}

// ---------------------------------------------------------------- leftovers
// The leading parts of a double-float matrix as an FP32 GEMM operand.
struct ViewHi {
  const dfl* p;
  int ld;
  __device__ __forceinline__ float get(int r, int c) const { return p[(size_t)r * ld + c].h; }
  __device__ __forceinline__ bool row_major() const { return true; }
};
// P = Gh (Y S~) + (S~ Y) Gh + G0 (Y Sh) + (Sh Y) G0 (see solve_mixed.cu) of the pairs whose fragment asks for it.
__global__ void __launch_bounds__(NT) k_mx_leftover(const OzPair* __restrict__ pairs, const MxPair* __restrict__ mp,
                                                    int n_pairs, const int* __restrict__ done,
                                                    const int* __restrict__ refresh, int max_r, float* scratch) {
  __shared__ float fsm[GEMM_SMEM_F32];
  float* A1 = scratch + (size_t)blockIdx.x * 2 * max_r * max_r;
  float* A2 = A1 + (size_t)max_r * max_r;
  for (int q = blockIdx.x; q < n_pairs; q += gridDim.x) {
    const OzPair p = pairs[q];
    if (done[p.frag] || !refresh[p.frag]) continue;
    const MxPair x = mp[q];
    const int r = p.r;
    const ViewHi Y{reinterpret_cast<const dfl*>(p.Y), r};
    cta_gemm_f32s<float>(r, r, r, 1.0, Y, ViewF{x.Sh, r, 0}, 0.0, A1, r, fsm);
    cta_gemm_f32s<float>(r, r, r, 1.0, ViewF{x.Sh, r, 0}, Y, 0.0, A2, r, fsm);
    for (int idx = threadIdx.x; idx < r * r; idx += NT) {
      const int a = idx / r, b = idx % r;
      const float y = Y.get(a, b);
      x.P[idx] = (float)(p.et[a] - 0.5 * p.fij) * A1[idx] + (float)(p.et[b] - 0.5 * p.fij) * A2[idx];
      A1[idx] += y;
      A2[idx] += y;
    }
    __syncthreads();
    cta_gemm_f32s<float>(r, r, r, 1.0, ViewF{x.Gh, r, 0}, ViewF{A1, r, 0}, 1.0, x.P, r, fsm);
    cta_gemm_f32s<float>(r, r, r, 1.0, ViewF{A2, r, 0}, ViewF{x.Gh, r, 0}, 1.0, x.P, r, fsm);
  }
}

// ---------------------------------------------------------------- update
constexpr int MXT = 512, MU = 4;
// Bound: HBM, 36 bytes an element read, 8 written and 8 a version of digits (2.9 ms at 160 million elements); four
// elements a thread in flight (19 ms without).  Y stays in shared memory (cap pairs) for the transposed reads.
__global__ void __launch_bounds__(MXT) k_mx_update(const OzPair* __restrict__ pairs, const MxPair* __restrict__ mp,
                                                  int n_pairs, const int* __restrict__ done, int first, int ld, size_t slice,
                                                  int cap, uint16_t* __restrict__ D, int* __restrict__ ex,
                                                  int* __restrict__ exW, double* __restrict__ pe,
                                                  double* __restrict__ pu) {
  extern __shared__ dfl ysm[];
  __shared__ float red[4][MXT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = blockIdx.x; q < n_pairs; q += gridDim.x) {
    const OzPair p = pairs[q];
    if (done[p.frag]) continue;
    const MxPair x = mp[q];
    const int r = p.r, pitch = r | 1;
    const bool in = r * pitch <= cap;
    dfl* Y = reinterpret_cast<dfl*>(p.Y);
    const dfl* C = reinterpret_cast<const dfl*>(p.C);
    dfl* Ys = in ? ysm : Y;
    const int ys = in ? pitch : r;
    const unsigned rr = (unsigned)(r * r), mag = row_magic((unsigned)r);
    float du = 0.f, am = 0.f, ss = 0.f;
    float sh = 0.f, sl = 0.f;              // <K~, 2 Y>
    for (unsigned i0 = threadIdx.x; i0 < rr; i0 += MU * MXT) {   // MU elements' loads in flight
      dfl kd[MU], id[MU], c[MU], yo[MU];
      float pp[MU];
#pragma unroll
      for (int u = 0; u < MU; u++) {
        const unsigned idx = min(i0 + u * MXT, rr - 1);
        kd[u] = x.Kd[idx];
        id[u] = x.iD[idx];
        if (!first) {
          c[u] = C[idx];
          pp[u] = x.P[idx];
          yo[u] = Y[idx];
        } else {
          c[u] = yo[u] = dfl{0.f, 0.f};
          pp[u] = 0.f;
        }
      }
#pragma unroll
      for (int u = 0; u < MU; u++) {
        const unsigned idx = i0 + u * MXT;
        if (idx >= rr) break;
        const dfl y = df_mul(df_add(kd[u], df_add(c[u], dfl{pp[u], 0.f})), id[u]);
        const float d = fabsf((y.h - yo[u].h) + (y.l - yo[u].l));
        du = d <= du ? du : d;             // a NaN stays
        am = fmaxf(am, fabsf(y.h));
        ss = fmaf(y.h, y.h, ss);
        df_acc(sh, sl, kd[u], dfl{2.f * y.h, 2.f * y.l});
        Y[idx] = y;
        if (in) {
          const unsigned a = row_of(idx, (unsigned)r, mag);
          ysm[a * pitch + (idx - a * r)] = y;
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float d = __shfl_xor_sync(0xffffffffu, du, o);
      du = d <= du ? du : d;
      am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
      ss += __shfl_xor_sync(0xffffffffu, ss, o);
    }
    if (lane == 0) {
      red[0][warp] = du;
      red[1][warp] = am;
      red[2][warp] = ss;
    }
    __syncthreads();                       // Y is complete
    du = red[0][0];
    am = red[1][0];
    ss = red[2][0];
#pragma unroll
    for (int u = 1; u < MXT / 32; u++) {
      du = red[0][u] <= du ? du : red[0][u];
      am = fmaxf(am, red[1][u]);
      ss += red[2][u];
    }
    const bool bad = !isfinite(ss) || !isfinite(du);
    for (unsigned i0 = threadIdx.x; i0 < rr; i0 += MU * MXT) {   // -<K~, Y^T>
      dfl kd[MU];
#pragma unroll
      for (int u = 0; u < MU; u++) kd[u] = x.Kd[min(i0 + u * MXT, rr - 1)];
#pragma unroll
      for (int u = 0; u < MU; u++) {
        const unsigned idx = i0 + u * MXT;
        if (idx >= rr) break;
        const unsigned a = row_of(idx, (unsigned)r, mag);
        df_acc(sh, sl, kd[u], df_neg(Ys[(idx - a * r) * ys + a]));
      }
    }
    dfl e = df_norm(sh, sl);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e = df_add(e, df_shfl_xor(e, o));
    __syncthreads();
    if (lane == 0) {
      red[0][warp] = e.h;
      red[1][warp] = e.l;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      dfl s{red[0][0], red[1][0]};
      for (int u = 1; u < MXT / 32; u++) s = df_add(s, dfl{red[0][u], red[1][u]});
      const double ed = df_to(s);
      pe[q] = p.diag ? ed : 2.0 * ed;
      pu[q] = bad ? __longlong_as_double(0x7FF8000000000000ll) : (double)du;
    }
    const int eY = bad ? oz::EX_ZERO : exp_code(am), eW = bad ? oz::EX_ZERO : exp_code(sqrtf(ss) * 1.001f);
    for (int v = 0; v < 3; v++) {
      const int id = p.ver[v];
      if (id < 0) continue;
      const int up = v == 2, ey = live_code(eY) ? eY + up : eY, ew = live_code(eW) ? eW + up : eW;
      if (threadIdx.x == 0) {
        ex[id] = ey;
        exW[id] = ew;
      }
      uint16_t* base = D + (size_t)p.vrow[v] * ld;
      for (int m = warp; m < r; m += MXT / 32) {
        uint16_t* dst = base + (size_t)m * ld;
        if (v == 0) row_digits([&](int k) { return Ys[m * ys + k]; }, r, 0, p.kpad, ey, dst, slice);
        else if (v == 1) row_digits([&](int k) { return Ys[k * ys + m]; }, r, 0, p.kpad, ey, dst, slice);
        else row_digits([&](int k) { return df_add(Ys[m * ys + k], Ys[k * ys + m]); }, r, 0, p.kpad, ey, dst, slice);
      }
    }
    __syncthreads();
  }
}

// One exponent code for the W of a pair's terms: the largest of Y's norm times the coefficient.
__global__ void k_mx_bounds(const int* __restrict__ term0, const MxBound* __restrict__ terms, int n_pairs,
                            const int* __restrict__ exW, int* __restrict__ eP) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n_pairs) return;
  int e = oz::EX_ZERO;
  for (int t = term0[p]; t < term0[p + 1]; t++) {
    const int x = exW[terms[t].ver];
    if (x > oz::EX_ZERO / 2) e = max(e, x + terms[t].e);
  }
  eP[p] = e;
}

// As k_oz_converge, and when P of a fragment is to be formed again: after a move of more than P_LAG of the scale of
// its amplitudes since it was last formed.
constexpr double P_LAG = 1e-2;
__global__ void k_mx_converge(const int* __restrict__ pair0, int n_frag, const double* __restrict__ pe,
                              const double* __restrict__ pu, SolveOpts o, int it, double* __restrict__ e_prev,
                              double* __restrict__ scale, double* __restrict__ drift, int* __restrict__ refresh,
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
  else if (um < o.tol_update && fabs(e - e_prev[f]) < fmax(o.tol_energy, 1e-11 * fabs(e))) status = 0;
  e_prev[f] = e;
  if (it == 1) scale[f] = um;
  const double dr = drift[f] + um;
  const bool again = dr > P_LAG * scale[f];
  refresh[f] = again;
  drift[f] = again ? 0.0 : dr;
  out[out_id[f]] = FragOut{e, nan ? __longlong_as_double(0x7FF8000000000000ll) : um, it, status};
  if (status != ERR_NOCONV || it == o.max_iter) done[f] = 1;
  else atomicAdd(left, 1);
}

// Y to FP64, into the slots of the gradient.
__global__ void __launch_bounds__(NT) k_mx_store(const OzPair* __restrict__ pairs) {
  const OzPair p = pairs[blockIdx.x];
  const dfl* Y = reinterpret_cast<const dfl*>(p.Y);
  for (int idx = threadIdx.x; idx < p.r * p.r; idx += NT) p.T[idx] = df_to(Y[idx]);
}

int mx_cap(int max_r, size_t elem) {       // elements of dynamic shared memory for one padded matrix
  const size_t need = (size_t)max_r * (max_r | 1) * elem;
  return (int)(std::min<size_t>(need, 200 * 1024) / elem);
}

}  // namespace

void launch_mx_sigma(const MxSigma* jobs, int n, int max_r, int ld, long long rows, uint16_t* D, int n_cta,
                     cudaStream_t st) {
  if (!n) return;
  const int cap = mx_cap(max_r, sizeof(float));
  allow_dynamic_smem((const void*)k_mx_sigma);
  k_mx_sigma<<<std::min(n, n_cta), NT, cap * sizeof(float), st>>>(jobs, n, ld, (size_t)rows * ld, cap, D);
  note_launch(1);
}
void launch_mx_bounds(const int* term0, const MxBound* terms, int n_pairs, const int* exW, int* eP, cudaStream_t st) {
  if (!n_pairs) return;
  k_mx_bounds<<<(n_pairs + 127) / 128, 128, 0, st>>>(term0, terms, n_pairs, exW, eP);
  note_launch(1);
}
void launch_mx_tables(const MxTable* jobs, int n, cudaStream_t st) {
  if (!n) return;
  k_mx_tables<<<dim3(n, 4), NT, 0, st>>>(jobs);
  note_launch(1);
}
void launch_mx_leftover(const OzPair* pairs, const MxPair* mp, int n, const int* done, const int* refresh, int max_r,
                        float* scratch, int n_cta, cudaStream_t st) {
  if (!n) return;
  k_mx_leftover<<<n_cta, NT, 0, st>>>(pairs, mp, n, done, refresh, max_r, scratch);
  note_launch(1);
}
void launch_mx_update(const OzPair* pairs, const MxPair* mp, int n, const int* done, bool first, int max_r, int ld,
                      long long rows, uint16_t* D, int* ex, int* exW, double* pe, double* pu, int n_cta, cudaStream_t st) {
  if (!n) return;
  const int cap = mx_cap(max_r, sizeof(dfl));
  allow_dynamic_smem((const void*)k_mx_update);
  k_mx_update<<<n_cta, MXT, cap * sizeof(dfl), st>>>(pairs, mp, n, done, first ? 1 : 0, ld, (size_t)rows * ld, cap, D, ex, exW,
                                                             pe, pu);
  note_launch(1);
}
void launch_mx_converge(const int* pair0, int n_frag, const double* pe, const double* pu, SolveOpts o, int it,
                        double* e_prev, double* scale, double* drift, int* refresh, int* done, int* left, FragOut* out,
                        const int* out_id, cudaStream_t st) {
  if (!n_frag) return;
  cudaMemsetAsync(left, 0, sizeof(int), st);
  k_mx_converge<<<(n_frag + 127) / 128, 128, 0, st>>>(pair0, n_frag, pe, pu, o, it, e_prev, scale, drift, refresh, done,
                                                      left, out, out_id);
  note_launch(1);
}
void launch_mx_store(const OzPair* pairs, int n, cudaStream_t st) {
  if (!n) return;
  k_mx_store<<<n, NT, 0, st>>>(pairs);
  note_launch(1);
}

}  // namespace osv

// Internal interfaces between the host runtime (api.cu) and the kernel
// translation units of libosvmp2.  Not part of the C ABI.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include "common.cuh"
#include "oz_job.h"
#include "tc_job.h"

namespace osv {

// Device-resident lookup tables of the pair store (all pointers are device).
struct Tables {
  int n_occ;
  int n_vir;
  const int* n_osv;             // [n_occ]
  const double* const* Q;       // [n_occ] -> Q_i [n_vir][n_osv_i]
  const int* sf_id;             // [n_occ*n_occ]: (x<=y) -> S/F block id, -1 if absent
  const double* const* S;       // [n_blocks] S_(x,y) [n_x][n_y]
  const double* const* F;       // [n_blocks] F_(x,y)
  const int* pair_id;           // [n_occ*n_occ]: (i<=j) -> pair id, -1 if absent
  const double* const* K;       // [n_pairs] K_(ij,ij) [m][m]
  const double* const* X;       // [n_pairs] X [m][m] (first r columns valid)
  const double* const* et;      // [n_pairs] e~ [m] (first r valid)
  const int* r;                 // [n_pairs]
  const double* const* Kt;      // [n_pairs] K~ = X^T K X  [r][r]
  const float* const* U;        // [n_pairs] mixed form: U = P X  [n_vir][r] (FP32)
  const float* const* Sh;       // [n_pairs] mixed form: X^T S X - 1 [r][r] (FP32), NULL if X is exact
  const float* const* Gh;       // [n_pairs] mixed form: X^T F X - diag(e~) - (f_ii+f_jj)/2 Sh [r][r]
  const double* f_occ;          // [n_occ][n_occ]
};

// Process-wide count of kernel launches issued by the library.
void note_launch(int n);

// Lets kernel fn ask for all the dynamic shared memory that its static part leaves of a CTA's 227 KB.  The limit belongs
// to the process, so it is this one in every call: set to the size of the call at hand, another thread's smaller
// system could lower it before the launch.
inline cudaError_t allow_dynamic_smem(const void* fn) {
  cudaFuncAttributes a;
  const cudaError_t e = cudaFuncGetAttributes(&a, fn);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024 - (int)a.sharedSizeBytes);
}

struct SolveOpts {
  double tol_update, tol_energy;
  int max_iter;
  int tiles;      // mixed solver: tile set of its FP32 contractions (cta_gemm_f32s)
};

// Per-fragment result record written by the solvers.
struct FragOut {
  double energy;
  double umax;
  int iters;
  int status;   // 0 ok, ERR_* bits otherwise
};

// ---- A0 (osv_build.cu)
// T_ii of orbitals [i0, i0+nb) into T [nb][nv][nv].
void launch_tii(const BSrc& src, const double* e_vir, const double* f_occ, int n_occ, int i0, int nb,
                double* T, cudaStream_t st);
// Eigen-decomposition of each T[b] and selection omega >= thr (all if thr <= 0),
// at most kmax per orbital: V [nb][kmax][nv] (eigenvector-major), w [nb][kmax], k [nb], err |= ERR_*.
// nclu: eig_cluster_table.
// Per-orbital scratch: d, e, tau (3 nv); the work room (exchange buffers of the tridiagonalisation, Z of a
// full decomposition, 4 or more groups x 176 nv of lane-batched inverse iteration, the Gram matrix
// of the kept vectors); the kept vectors of the tridiagonal.
__host__ __device__ inline size_t eig_osv_work_doubles(int nv) {
  return (size_t)nv * nv > (size_t)4 * 176 * nv ? (size_t)nv * nv : (size_t)4 * 176 * nv;
}
__host__ __device__ inline size_t eig_osv_scratch_doubles(int nv, int kmax) {
  return (size_t)3 * nv + eig_osv_work_doubles(nv) + (size_t)kmax * nv + 64;
}
// dfl_tridiag: the top-k path tridiagonalises in double-float arithmetic (the
// mixed-form OSV build, whose T_ii is a split-precision product).
void launch_eig_osv(double* T, int nb, int nv, double thr, int kmax, double* V, double* w, int* k,
                    double* scratch, int* err, bool dfl_tridiag, const int* nclu, cudaStream_t st,
                    cudaStream_t st_qr = nullptr, cudaEvent_t fork = nullptr);   // fork: the implicit QR on st_qr, after st so far
// Back-transformation of the kept eigenvectors of the top-k path (n_vir above
// the shared-memory limit, thr > 0) after launch_eig_osv; a no-op otherwise.
void launch_eig_back(double* T, int nb, int nv, double thr, int kmax, double* V, const int* k, double* scratch,
                     bool dfl_tridiag, cudaStream_t st);
// Randomized OSVs (rosv.cu; Algorithm 3) for a batch of nb orbitals with T_ii in
// T [nb][nv][nv].  Scratch layout (offsets in doubles) from rosv_layout; the
// Gaussian draw k of orbital i, entry a, is the Irwin-Hall normal of counter
// (i * ROSV_ROWS_PER_ORBITAL + k) * nv + a on the key of stream 7 of the seed.
constexpr uint64_t ROSV_ROWS_PER_ORBITAL = 1ull << 16;
constexpr int ROSV_WINDOW = 10;   // look-ahead rows r of the range finder
struct RosvLayout {
  int rows;                 // r + n_max Gaussian rows per orbital
  size_t y, z, tt, svd, svd_per, wmax, nrows, total;
  int ldk;                  // row stride of the TF32 slice store (mixed form)
  long long store_rows;     // rows of the slice store: nb * NSL * (nv + rows)
};
RosvLayout rosv_layout(int nb, int nv, int r, int n_max, int kmax);
// FP64 form: out[u] = A_u T_u with A_u the Gaussian rows (mode 0, rows rows) or
// Z_u (mode 1, nrows[u] of n_max = rows rows).
void launch_rosv_gemm64(int mode, const double* T, int nb, int nv, int i0, uint64_t key, const double* Z,
                        const int* nrows, int rows, double* out, cudaStream_t st);
// Mixed form: TF32 slices (K = nv) of T rows (part 0), Gaussian rows (1) or Z rows (2).
void launch_rosv_slices(int part, const double* T, int nb, int nv, int i0, uint64_t key, const double* Z,
                        int z_rows, const int* nrows, int rows, float* slices, int ldk, cudaStream_t st);
void launch_rosv_finder(double* Y, int nb, int nv, int r, int n_max, double l_osv, double* Z, int* nrows,
                        double* wmax, int* err, cudaStream_t st);
// FP64 form: M[u] = T~ T~^T ([nb][ldm][ldm], zero outside nrows[u]).
void launch_rosv_gram64(const double* Tt, const int* nrows, int nb, int nv, int n_max, int ldm, double* M,
                        cudaStream_t st);
// Q = Q~^T Z and omega = sqrt(eigenvalues of M) for the ks[u] kept eigenvectors Vs ([nb][ldm][ldm]).
void launch_rosv_backq(const double* Vs, const double* ws, const int* ks, const double* Z, const int* nrows, int nb,
                       int nv, int n_max, int ldm, int kmax, double* V, double* w, int* k, cudaStream_t st);
// Copy V[b][:, :k_b] into the packed Q store (Q[i0+b] as [nv][k]).
void launch_pack_q(const double* V, const double* w, int nb, int nv, int kmax, const int* k,
                   double* const* Qdst, double* const* wdst, cudaStream_t st);

// ---- FP64 contractions on the tensor cores (oz_gemm.cu, tc_oz.cuh)
// Digit store of an operand: per slice `rows` rows of K BF16 digits with stride ld (a multiple of 8), and chunk exponents.
struct OzOperand {
  const uint16_t* D;
  long long rows;
  int K, ld;
  const int* ex;
};
struct OzMat {           // dense matrix whose digits go to m; row stride ldm (see launch_oz_mats)
  const double* p;
  int rows, K, kpad, ldm;  // kpad >= K: digits of k in [K, kpad) are written as zeros
  oz::Mat m;
};
// ns: slices (NSL: FP64; MXSL: 39 bits, mixed form).
// Digits of B: rows B[i0 + u][a][.] (K = aux) or B[xs[u]][.][P] (K = vir); slot u, row r at row u rows + r of a store
// of nb rows per slice.
void launch_oz_rows(const BSrc& src, int i0, int nb, int ns, uint16_t* D, int* ex, cudaStream_t st);
void launch_oz_cols(const BSrc& src, const int* xs, int nb, int ns, uint16_t* D, int* ex, cudaStream_t st);
// Digits of dense matrices into a store of `rows` rows: [K][rows] (row index innermost), scaled by w[k] unless
// NULL; or, k_inner, [rows][K].
void launch_oz_mats(const OzMat* mats, int n, int max_rows, int max_K, const double* w, bool k_inner, int ns, int ld,
                    long long rows, uint16_t* D, int* ex, cudaStream_t st);
// out[row][col] per job (row-major); T_ii tiles of the lower triangle (mirrored, with denominators).
// Return 0, or -1 if a tensor map could not be encoded.
int launch_oz_gemm(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                   const int* skip, int* err, cudaStream_t st);
int launch_oz_tii(const OzOperand& A, const oz::Job* jobs, int n_jobs, const oz::Seg* segs, const double* e_vir, int ns,
                  int* err, cudaStream_t st);
// The digits of the output (jobs' o_row, o_e) into the store D of `rows` rows with stride ld (a multiple of 32).
int launch_oz_digits(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                     const int* skip, uint16_t* D, int ld, long long rows, const int* exW, int* err, cudaStream_t st);
// Dot products of (2 Y - Y^T) with the product of every job (see OzEpiDot), 16 partial sums per job.
int launch_oz_dots(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                   double* parts, int* err, cudaStream_t st);
// Sums of the squares of the product of every job (see OzEpiSquares), 16 partial sums per job.
int launch_oz_squares(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                      double* parts, int* err, cudaStream_t st);
// ---- FP64 amplitude iterations on the tensor cores (solve_oz.cu)
struct OzPolish {        // pair basis refinement
  int r, pad;
  const double* S1;      // U0^T U0 [r][r]
  double* F1;            // U0^T e U0 (overwritten)
  double* IE;            // out: the change of basis, U = U0 IE [r][r]
  double* et;            // out
  int* ok;               // out: this step was the last one the basis needed
};
void launch_oz_polish(const OzPolish* jobs, int n_jobs, int max_r, double* scratch, int n_cta, cudaStream_t st);
struct OzPair {          // a pair of a fragment
  int frag, r, m, diag;
  int kpad;              // r rounded up to 32
  int ver[3];            // matrix id of the digits of Y, Y^T, Y + Y^T, -1 where no term uses them
  int vrow[3];           // their store rows
  int pad;
  double fij;            // f_ii + f_jj
  const double* Kt;      // [r][r]
  const double* iD;      // 1 / D [r][r] (FP64 form)
  const double* et;      // [r]
  const double* X;       // [m][m]
  double* Y;             // [r][r]
  double* C;             // [r][r]
  double* T;             // [m][m] raw-basis amplitude (launch_oz_raw) or NULL
};
void launch_oz_update(const OzPair* pairs, int n_pairs, const int* done, bool first, int ld, long long rows, int nch, uint16_t* D,
                      int* ex, int* exW, double* pe, double* pu, int n_cta, cudaStream_t st);
struct OzTable {         // iD of a pair: 1 / (fij - e_a - e_b)
  int r, pad;
  double fij;
  const double* et;
  double* iD;
};
void launch_oz_tables(const OzTable* jobs, int n, cudaStream_t st);
void launch_oz_converge(const int* pair0, int n_frag, const double* pe, const double* pu, SolveOpts o, double ulps, int it,
                        double* e_prev, int* done, int* left, FragOut* out, const int* out_id, cudaStream_t st);
void launch_oz_raw(const OzPair* pairs, int n_pairs, int max_m, double* scratch, int n_cta, cudaStream_t st);
// Mixed form (solve_mx.cu): Y and C are double-float pairs in the same storage, coef of a segment the bits of a pair.
struct MxPair {          // beside OzPair
  const dfl* Kd;         // K~ and 1 / D [r][r]
  const dfl* iD;
  const float* Sh;
  const float* Gh;
  float* P;              // [r][r], zero until first formed
};
struct MxSigma {         // digits of S (rl x rh) and of its transpose
  const float* S;
  int rl, rh;
  oz::Mat lo, hi;
};
struct MxTable {
  int r, pad;
  double fij;
  const double* Kt;
  const double* et;
  dfl* Kd;
  dfl* iD;
};
void launch_mx_sigma(const MxSigma* jobs, int n, int max_r, int ld, long long rows, uint16_t* D, int n_cta,
                     cudaStream_t st);
void launch_mx_tables(const MxTable* jobs, int n, cudaStream_t st);
void launch_mx_leftover(const OzPair* pairs, const MxPair* mp, int n, const int* done, const int* refresh, int max_r,
                        float* scratch, int n_cta, cudaStream_t st);
void launch_mx_update(const OzPair* pairs, const MxPair* mp, int n, const int* done, bool first, int max_r, int ld,
                      long long rows, uint16_t* D, int* ex, int* exW, double* pe, double* pu, int n_cta,
                      cudaStream_t st);
void launch_mx_converge(const int* pair0, int n_frag, const double* pe, const double* pu, SolveOpts o, int it,
                        double* e_prev, double* scale, double* drift, int* refresh, int* done, int* left, FragOut* out,
                        const int* out_id, cudaStream_t st);
void launch_mx_store(const OzPair* pairs, int n, cudaStream_t st);
// W digits under the codes eP of the pairs (job.o_e; Y's code eY[job.ld_out], coefficient job.s), and C from them.
int launch_mx_w(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                const int* skip, uint16_t* D, int ld, long long rows, const int* eY, const int* eP, int* err,
                cudaStream_t st);
int launch_mx_c(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                const int* skip, const int* eP, int* err, cudaStream_t st);
struct MxBound {         // a term of a pair: id of its Y matrix, exponent of its coefficient (|c| < 2^e)
  int ver, e;
};
void launch_mx_bounds(const int* term0, const MxBound* terms, int n_pairs, const int* exW, int* eP, cudaStream_t st);
struct OzDf {            // dE/df of a fragment of nc <= 3 orbitals
  int nc, pair0, out;    // its pairs; fragment index of the result
  int pad;
  double weight;
  int tile0[10];         // tiles of dot t: [tile0[t], tile0[t + 1])
};
void launch_oz_df(const OzDf* frags, int n_frag, const OzPair* pairs, const double* parts, double* g, int n_cta,
                  cudaStream_t st);
struct OzGradPair {      // adjoint of a pair
  int r, m, c0, c1;      // contributions [c0, c1) (Y of a fragment, its weight)
  const double* X;
  double *Wy, *Hy;       // [r][r]
  double *W, *H;         // [m][m] raw basis
};
struct GradContrib;
void launch_oz_gsum(const OzGradPair* jobs, int n_jobs, const GradContrib* con, cudaStream_t st);
void launch_oz_graw(const OzGradPair* jobs, int n_jobs, int max_m, double* scratch, int n_cta, cudaStream_t st);
// cuTensorMapEncodeTiled (NULL if the driver has none)
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder();

// ---- A1-A2 (pair_integrals.cu)
struct ProjJob {         // B~_{i}^{(x)} = B[i]^T Q_x  -> out [n_aux][n_x]
  int i, x;
  double* out;
};
void launch_project(const BSrc& src, const Tables& t, const ProjJob* jobs, int n_jobs, int max_nx, int fp32,
                    cudaStream_t st);
struct KJob {            // K_(ij,ij) from the projections
  int i, j;
  const double* Bii;     // B~_i^(i)  [n_aux][n_i]
  const double* Bij;     // B~_i^(j)  [n_aux][n_j]   (NULL if i == j)
  const double* Bji;     // B~_j^(i)
  const double* Bjj;     // B~_j^(j)
  double* out;           // [m][m]
};
void launch_exchange(const Tables& t, int n_aux, const KJob* jobs, int n_jobs, int max_m, int fp32, cudaStream_t st);
struct SFJob {           // S_(x,y), F_(x,y)
  int x, y;
  double* S;
  double* F;
};
void launch_sf(const Tables& t, const double* e_vir, const SFJob* jobs, int n_jobs, int max_n,
               cudaStream_t st);

// ---- A3 (precond.cu)
struct PJob {            // preconditioner of pair (i,j): X, e~, r (+ the mixed form's leftovers)
  int i, j;
  double* X;
  double* et;
  int* r;
  float* Sh;             // mixed form only: X^T S X - 1          [r][r]
  float* Gh;             // mixed form only: X^T F X - diag(e~) - (f_ii+f_jj)/2 Sh
};
__host__ __device__ inline size_t precond_scratch_doubles(int max_m) {
  return 6 * (size_t)max_m * max_m + 4 * (size_t)max_m + 64;
}
void launch_precond(const Tables& t, double tau_s, const PJob* jobs, int n_jobs, int max_m, double* scratch,
                    int n_cta, int* err, cudaStream_t st);
// out = Xc (Xc^T S X) of the pair (i, j), W: 2 m r doubles.
void launch_precond_rewrite(const Tables& t, int i, int j, const double* Xc, const double* X, int r, double* W,
                            double* out, cudaStream_t st);
// One warp per pair (pair order <= 192); returns -1 if max_m is too large.
size_t precond_w_scratch_doubles(int max_m, int n_warps);
int launch_precond_w(const Tables& t, double tau_s, const PJob* jobs, int n_jobs, int max_m, double* scratch,
                     int n_warps, int* err, cudaStream_t st);
// precond_mixed.cu: block-structured orthogonalisation in FP64, F' diagonalised in FP32, with exact
// leftovers Sh/Gh for the jobs that have them (mixed form; in the FP64 form the basis is polished
// afterwards); max_n: the largest OSV count; -1 if max_m is too large.
// Per-pair intermediates: one slot of precond_mixed_slot_doubles(m) at slots + off[job];
// mdim[job] = pair order m; order: the jobs in the order the CTAs take them
// (grid-stride; descending m balances the launch).
size_t precond_mixed_slot_doubles(int m);
size_t precond_mixed_scratch_doubles(int max_m, int n_cta);
int launch_precond_mixed(const Tables& t, double tau_s, const PJob* jobs, const int* order, int n_jobs, int max_m, int max_n,
                         const int* m_sorted, double* slots, const long long* off, const int* mdim, double* scratch,
                         int n_cta, int num_sms, int* err, cudaStream_t st);

// ---- A4-A5 (solve.cu)
// Fragments: orbs [n][3] (-1 padded, ascending), order[] = processing order.
// per CTA: T, R, G1, G2 for six pairs + two work matrices
__host__ __device__ inline size_t frag_scratch_doubles(int max_m) { return 26 * (size_t)max_m * max_m + 64; }
// Tstore (may be NULL): converged amplitudes of fragment f are written at
// Tstore + Toff[f], local pairs (a<=b) in order, each m_p x m_p.
void launch_frag_solve(const Tables& t, const int* frag_orbs, const int* order, int n_frag, int max_m,
                       SolveOpts o, double* scratch, int n_cta, int* counter, FragOut* out,
                       double* Tstore, const long long* Toff, cudaStream_t st);
// Mixed-form pair build in the orthonormal pair basis U = P X: contractions of MXSL slices, summed as FP32 pairs.
// G = U^T B per job (A rows: aux, B rows: pair basis): out[col][row] of leading parts, remainders lo_shift floats on.
int launch_mx_g(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                long long lo_shift, int* err, cudaStream_t st);
// out[row][col] in FP64 or FP32
int launch_mx_gemm(const OzOperand& A, const OzOperand& B, const oz::Job* jobs, int n_jobs, const oz::Seg* segs,
                   bool fp64_out, int* err, cudaStream_t st);
// Digits of matrices of FP32 pairs (OzMat.p: the leading parts, [rows][K]).
void launch_mx_pairs(const OzMat* mats, int n, int max_rows, int K, long long lo_shift, int ld, long long rows,
                     uint16_t* D, int* ex, cudaStream_t st);
void launch_oz_float(const double* x, size_t n, float* y, cudaStream_t st);
// Products of TF32 slice rows (randomized OSVs): Gs holds `rows` rows of K = n_aux, FP64 row-major output.
int launch_kt_tc(const float* Gs, long long rows, int n_aux, int ldg, const tc::Job* jobs, int n_jobs, int* err,
                 cudaStream_t st);
// 2-D FP32 tensor map over rows x n_k (row stride ldk floats, a multiple of 4),
// 128-byte swizzle, box tc::BK x box_rows; false if the driver rejects it.
bool make_slice_map(CUtensorMap* m, const float* base, int n_k, int ldk, long long rows, int box_rows);

// Mixed form (solve_mixed.cu): per pair K~ = X^T K X, then the fragment solve in
// the preconditioner basis with FP32 coupling products.
struct KtJob {
  int i, j;
  double* Kt;
};
void launch_ktilde(const Tables& t, const KtJob* jobs, int n_jobs, double* scratch, int n_cta, int max_m,
                   cudaStream_t st);
// per CTA: Y, 1/D (6 + 6 FP64), C as (hi, lo) (12 FP32) + Y32 (6 FP32) + 3 work (FP32) + G0 (6 max_m FP32)
__host__ __device__ inline size_t frag_mixed_scratch_doubles(int max_m) {
  const size_t M2 = (size_t)max_m * max_m;
  return 24 * M2 + (15 * M2 + 6 * (size_t)max_m + 1) / 2 + 64;
}
// Pair-couple overlaps Sigma_(lo,hi) = U_lo^T U_hi (pair ids lo < hi) of one MBE
// call, stored [r_lo][r_hi] at base + pos[id]; the ids of couples (lo, *) are
// off[lo] .. off[lo+1]-1 with partner hi[id] ascending.
struct SigmaTable {
  const int* off;
  const int* hi;
  const long long* pos;
  const float* base;
};
void launch_frag_solve_mixed(const Tables& t, const int* frag_orbs, const int* order, int n_frag, int max_m,
                             SolveOpts o, const SigmaTable& sgt, double* scratch, int n_cta, int* counter,
                             FragOut* out, double* Tstore, const long long* Toff, int* err, int ctas_per_sm,
                             cudaStream_t st);
// E = sum_f w_f * E_f in a fixed order -> e_out (device scalar)
void launch_weighted_sum(const FragOut* out, const int* weights, int n, double* e_out, cudaStream_t st);

// General subsystem solve: one kernel per Jacobi sweep over pairs.
struct SubDev {
  int nc;
  const int* orbs;          // [nc]
  double* const* T;         // [np] amplitude per local pair
  double* const* R;         // [np]
  double* const* G1;        // [np] F_p - f_ii S_p
  double* const* G2;        // [np] F_p - f_jj S_p
  double* const* W;         // [n_cta] work matrices (2 per CTA: W, Rt)
  double* pe;               // [np] pair energies
  double* pu;               // [np] pair max|update|
};
void launch_sub_prepare(const Tables& t, const SubDev& s, int np, int n_cta, cudaStream_t st);
void launch_sub_residual(const Tables& t, const SubDev& s, int np, int n_cta, cudaStream_t st);
void launch_sub_update(const Tables& t, const SubDev& s, int np, int n_cta, cudaStream_t st);

// ---- A6 (grad.cu)
struct GradContrib {       // one fragment's amplitude of a pair and the fragment weight
  const double* T;
  int weight;
};

// ---- occupied-orbital localization (localize.cu; Algorithm 2)
// P: scratch [n][n][n_atom]; U out [n][n]; out[0] = L, out[1] = last dL; status[0] = sweeps,
// status[1] = 1 if converged (device).
void launch_pm_localize(const double* C, int n_ao, int n, const int* atom_ao, int n_atom, double l_loc, int max_sweeps,
                        double* P, double* U, double* out, int* status, int num_sms, cudaStream_t st);
// The same sweeps over a cooperative grid (atoms spread over the CTAs, one bounded grid
// barrier per step of disjoint rotations); false when the grid cannot be co-resident
// (nothing launched then).  P: n_atom n (n | 1) doubles; part: 4 * min(n_atom, num_sms) *
// (n / 2 + 1) doubles; bar: 2 unsigned; err |= ERR_TIMEOUT if a barrier wait gave up.
bool launch_pm_localize_grid(const double* C, int n, const int* atom_ao, int n_atom, double l_loc, int max_sweeps,
                             double* P, double* U, double* out, int* status, double* part, unsigned* bar, int* err,
                             int num_sms, cudaStream_t st);

// ---- pair screening and weak pairs (screen.cu), FP64 in both forms
// s2b[p] of the pairs (i, j) = pairs[p] (Eq. s2b), grid-stride over n_cta CTAs.
// s2b of a pair from the partial sums [tile0[p], tile0[p + 1]) of launch_oz_squares.
void launch_s2b_sum(const Tables& t, const int2* pairs, int n_pairs, const int* tile0, const double* parts, double* s2b,
                    cudaStream_t st);
void launch_s2b(const Tables& t, const int2* pairs, int n_pairs, double* s2b, int n_cta, cudaStream_t st);
struct DiagJob {           // T_ii (raw basis, [n_i][n_i]) = sum of contributions [c0, c1)
  int i, pid;              // orbital, id of the pair (i, i)
  int c0, c1;
  double* T;
};
// mixed != 0: contributions are Y (r x r) of the pair (i,i)'s preconditioner basis.
// scratch: 2 max_n^2 doubles per CTA.
void launch_diag_amp(const Tables& t, const DiagJob* jobs, int n_jobs, const GradContrib* contrib, int mixed,
                     double* scratch, int max_n, int n_cta, cudaStream_t st);
struct WeakJob {           // weak pair (i, j), i < j
  int i, j;
  const double* Bii;       // B~_i^(i) [n_aux][n_i]
  const double* Bjj;       // B~_j^(j) [n_aux][n_j]
  const double* S;         // S_(i,j) [n_i][n_j]
  const double* Ti;        // MBE(3) diagonal amplitude T_(i,i) [n_i][n_i]
  const double* Tj;
  const double* Xi;        // eigenbasis of F_(i,i) (columns; exact in the FP64 form, the mixed
  const double* Xj;        //   preconditioner basis of the pair (i,i) otherwise), row stride ldxi
  const double* ei;        // their eigenvalues
  const double* ej;
  int ldxi, ldxj;
  const double* Fi;        // F_(i,i) [n_i][n_i], F_(j,j) (mixed form's residual updates)
  const double* Fj;
};
// Weak-pair energies (both orders) into e_out[job]; scratch: 6 max_n^2 doubles per CTA.
void launch_weak(const Tables& t, int n_aux, const WeakJob* jobs, int n_jobs, double* scratch, int max_n, int n_cta,
                 double* e_out, int mixed, cudaStream_t st);
// Mixed form: B~_i^(i) = B_i^T Q_i in double-float for the jobs (i, x = i, out [n_aux][n_i]).
void launch_project_df(const BSrc& src, const Tables& t, const ProjJob* jobs, int n_jobs, cudaStream_t st);
struct GradPairJob {       // W_p = sum c T~, H_p = sum c (T~ S T^T + [i!=j] T~^T S T)
  int i, j;
  int c0, c1;              // contributions [c0, c1)
  double* W;
  double* H;
};
struct GradYTerm {         // rows [row0, row0+n_x) of W'_p (W or W^T) times P_p^T B_partner
  int pi, pj;
  int trans;
  int row0;
  const double* W;
  const double* Bt_i;      // B~_partner^(pi)  [n_aux][n_pi]
  const double* Bt_j;      // B~_partner^(pj)  [n_aux][n_pj]  (unused when pi == pj)
};
struct GradYJob {          // Y_o^(x) [n_x][n_aux] = sum of terms [t0, t1)
  int o, x;
  int t0, t1;
  double* Y;
};
struct GradBTerm {
  int x;
  const double* Y;
};
struct GradBJob {          // dB_i = 4 sum_x Q_x Y_i^(x) over terms [t0, t1)
  int i;
  int t0, t1;
};
void launch_grad_pair(const Tables& t, const GradPairJob* jobs, int n_jobs, const GradContrib* contrib,
                      double* scratch, int n_cta, int max_m, cudaStream_t st);
void launch_grad_de(const Tables& t, const GradPairJob* jobs, int n_jobs, double* scratch, int n_cta, int max_m,
                    double* dpair, double* de, cudaStream_t st);
void launch_grad_df(const Tables& t, const int* frag_orbs, const int* weights, const double* Tstore,
                    const long long* Toff, int n_frag, int max_m, double* scratch, int n_cta, double* gfrag,
                    const int* fptr, const int* flist, double* df, cudaStream_t st);
void launch_grad_Y(const Tables& t, int n_aux, const GradYJob* jobs, int n_jobs, const GradYTerm* terms, int max_n,
                   cudaStream_t st);
void launch_grad_dB(const Tables& t, int n_aux, const GradBJob* jobs, int n_jobs, const GradBTerm* terms, double* dB,
                    cudaStream_t st);

// ---- A6, OSV-relaxed part (grad_relax.cu)
struct RelaxKJob {          // exchange part of dP_(i,j): alpha [B_i (A_j W~^T) + B_j (A_i W~)]
  int i, j;
  const double* W;          // W~ = sum_C c_C T~ [m][m]
  const double* bt_ii;      // B_i^T Q_i [n_aux][n_i]
  const double* bt_ij;      // B_i^T Q_j (unused for i = j)
  const double* bt_ji;      // B_j^T Q_i
  const double* bt_jj;      // B_j^T Q_j
  double* out;              // [n_vir][m]: first term
  double* out2;             // second term; may be out (then added, by a launch of its own)
};
struct RelaxFragJob {       // the rest of dP for pairs [u0, u1) (a <= b in order) of one fragment
  int orbs[3];
  int no, u0, u1;
  double c;                 // fragment weight
  const double* T;          // the fragment's amplitudes, pairs (a <= b) in order
  double* slot[3];          // [n_vir][n_x] per orbital of the fragment; NULL where none of the pairs has it
};
struct RelaxGTerm {         // a block of columns added into G_x
  const double* p;
  int ld, col0;
};
struct RelaxGJob {          // G_x = dE/dQ_x [n_vir][n_x] = sum of terms [t0, t1)
  int x;
  int t0, t1;
  double* G;
};
struct RelaxRJob {          // eigenvector response of orbital x
  int x;
  const double* V;          // all eigenvectors of T_xx, eigenvector-major, descending eigenvalues
  const double* w;          // [n_vir] eigenvalues, descending
  const double* T;          // T_xx [n_vir][n_vir]
  const double* G;          // dE/dQ_x [n_vir][n_x]
  double* Z;                // [n_vir][n_vir]: the adjoint of T_xx, then Z / D
  double* Y;                // [n_vir - n_x][n_x]
  double* Xr;               // [n_vir][n_x]
  double* de;               // [n_vir]
  double* df;               // [1]
};
void launch_relax_kpart(const Tables& t, const BSrc& bs, const RelaxKJob* jobs, int n_jobs, double* scratch,
                        int n_cta, int max_m, bool both, cudaStream_t st);
void launch_relax_frag(const Tables& t, const double* e_vir, const RelaxFragJob* jobs, int n_jobs, double* scratch,
                       size_t scr_per, int n_cta, int max_m, int* next, cudaStream_t st);
void launch_relax_gather(int n_vir, const int* n_osv, const RelaxGJob* jobs, int n_jobs, const RelaxGTerm* terms,
                         cudaStream_t st);
void launch_relax_resp(const Tables& t, const BSrc& bs, const double* e_vir, const RelaxRJob* jobs, int nb,
                       double* dB, double* de, double* df, cudaStream_t st);
void launch_grad_de_reduce(const double* dpair, int n_pairs, int nv, double* de, cudaStream_t st);
void launch_grad_df_reduce(const Tables& t, const int* frag_orbs, const double* gfrag, int n_frag, const int* fptr,
                           const int* flist, double* df, cudaStream_t st);

// ---- A6, mixed form (grad_mixed.cu): Tstore holds Y_p (T_p = X_p Y_p X_p^T)
struct GradZJob {          // Z = op(W~) G  [r][n_aux]
  int r;
  int trans;
  const double* W;
  const float* G;
  float* Z;
};
struct GradMBTerm {        // U_p [n_vir][r] times Z [r][n_aux]
  int r;
  const float* U;
  const float* Z;
};
void launch_gradm_pair(const Tables& t, const GradPairJob* jobs, int n_jobs, const GradContrib* contrib,
                       double* scratch, int n_cta, int max_m, cudaStream_t st);
void launch_gradm_de(const Tables& t, const GradPairJob* jobs, int n_jobs, double* scratch, int n_cta, int max_m,
                     double* dpair, double* de, cudaStream_t st);
void launch_gradm_df(const Tables& t, const int* frag_orbs, const int* weights, const double* Tstore,
                     const long long* Toff, int n_frag, int max_m, double* scratch, int n_cta, double* gfrag,
                     const int* fptr, const int* flist, double* df, cudaStream_t st);
void launch_gradm_Z(int n_aux, const GradZJob* jobs, int n_jobs, int max_r, cudaStream_t st);
void launch_gradm_dB(int n_vir, int n_aux, const GradBJob* jobs, int n_jobs, const GradMBTerm* terms, double* dB,
                     cudaStream_t st);

}  // namespace osv

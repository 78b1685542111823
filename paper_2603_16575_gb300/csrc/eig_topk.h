// Cluster tridiagonalisation and eigenpairs above a threshold (eig_topk.cu).
#pragma once
#include <cuda_runtime.h>

namespace osv {

// Whether the vectors of a step and one warp's staging rows of the reduction fit shared memory (orders up to 9536);
// larger matrices must not be given to the calls below.
bool eig_order_fits(int n);
// nclu[C], C = 1..8: clusters of C CTAs of the tridiagonalisation that the GPU holds at a time.
void eig_cluster_table(int* nclu);
// T (nb matrices of order n >= 3, lower triangles): d, e, tau at the start of each matrix's scratch
// (eig_osv_scratch_doubles(n, kmax)), reflector k in row k to the right of the diagonal.
void launch_eig_tridiag(double* T, int nb, int n, int kmax, double* scratch, int* err, const int* nclu,
                        cudaStream_t st);
// As above, then the eigenvalues >= thr (w, descending, and their number k) and the eigenvectors of the
// tridiagonal (V, [k][n] per matrix).  df: double-float arithmetic; refl_df: reflectors stored as pairs.
void launch_eig_topk(double* T, int nb, int n, double thr, int kmax, double* V, double* w, int* k, double* scratch,
                     int* err, bool df, bool refl_df, const int* nclu, cudaStream_t st);

}  // namespace osv

// Split-TF32 tensor-core products of the randomized OSVs (tc_tf32x3.cuh), and the tensor maps.
#include "internal.h"
#include "tc_tf32x3.cuh"

namespace osv {

// out[row][col] = hi + lo in FP64 (row-major)
struct EpiRow64 {
  static constexpr bool kWarp = false;
  __device__ __forceinline__ void operator()(const tc::Job& jb, int r, int c, float h, float l) const {
    static_cast<double*>(jb.out)[(size_t)r * jb.ld_out + c] = (double)h + (double)l;
  }
};

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// 2-D FP32 map over rows x n_k (row stride ldk floats), 128-byte swizzle, box 32 x box_rows.
bool make_slice_map(CUtensorMap* m, const float* base, int n_k, int ldk, long long rows, int box_rows) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)n_k, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ldk * 4};
  cuuint32_t box[2] = {(cuuint32_t)tc::BK, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int launch_kt_tc(const float* Gs, long long rows, int n_aux, int ldg, const tc::Job* jobs, int n_jobs, int* err,
                 cudaStream_t st) {
  if (!n_jobs) return 0;
  if (cudaFuncSetAttribute(tc::k_tf32x3<EpiRow64>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::SMEM) !=
      cudaSuccess)
    return -1;
  CUtensorMap ma, mb;
  if (!make_slice_map(&ma, Gs, n_aux, ldg, rows, tc::BM) || !make_slice_map(&mb, Gs, n_aux, ldg, rows, tc::BROWS))
    return -1;
  tc::k_tf32x3<EpiRow64><<<tc::persistent_grid(n_jobs), tc::NTHREADS, tc::SMEM, st>>>(ma, mb, jobs, n_jobs, n_aux, err, EpiRow64{});
  note_launch(1);
  return 0;
}

}  // namespace osv

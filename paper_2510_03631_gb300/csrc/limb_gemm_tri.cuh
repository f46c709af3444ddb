// Launch interface of the three-limb CTA-pair tensor-core GEMM (limb_gemm_tri.cu).
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "vec_sums.cuh"

namespace qpadl {

// Limb rows per box of the vector operand: 32 vectors x 3 limbs.
constexpr uint32_t kTriGroup = 32;

// Where the sums of NV vectors lie behind their limbs: three fp16 rows of `pitch` each (then the sums end within
// 8 NV pitch bytes), or four byte limbs for limb_gemm_pair.cu and limb_gemm.cu (limb k of vector v in row 4 v + k).
// The GEMMs need the digits' centre beside them, the kernels that make them do not.
inline VecSums tri_sums(const __half *L, uint32_t nv, uint64_t pitch, uint32_t parts, uint32_t centre = 0) {
    return VecSums{reinterpret_cast<const uint32_t *>(L + 3ull * nv * pitch), nv, parts, centre};
}
inline VecSums four_sums(const __half *L, uint32_t nv, uint64_t pitch, uint32_t parts, uint32_t centre = 0) {
    return VecSums{reinterpret_cast<const uint32_t *>(L + 4ull * nv * pitch), nv, parts, centre};
}

cudaError_t prepare_limb_gemm_tri_kernels();

// Limbs (11, 11 and 10 bits, balanced) of NV vectors (vector v at X + v * x_ld) into L, limb k of
// vector v in row 3 v + k, and the vectors' sums behind them (limb_sum_parts(C) words each).  When `zero` is
// given, the same launch zeroes zero_words words there.
cudaError_t launch_vec_limbs_tri(const uint32_t *X, uint64_t x_ld, uint32_t NV, uint64_t C, __half *L, uint64_t pitch,
                                 uint32_t *zero, uint64_t zero_words, cudaStream_t stream);
cudaError_t launch_vec_limbs_four(const uint32_t *X, uint64_t x_ld, uint32_t NV, uint64_t C, __half *L, uint64_t pitch,
                                  uint32_t *zero, uint64_t zero_words, cudaStream_t stream);
// The three limbs, or four, of the columns of A (C x n row-major), and one sum each: vector k is column k.
cudaError_t launch_mat_col_limbs_tri(const uint32_t *A, uint64_t C, uint32_t n, __half *L, uint64_t pitch,
                                     uint32_t *zero, uint64_t zero_words, cudaStream_t stream);
cudaError_t launch_mat_col_limbs_four(const uint32_t *A, uint64_t C, uint32_t n, __half *L, uint64_t pitch,
                                      cudaStream_t stream);

// How a product of these sizes is cut: 64-vector halves per tile, column ranges per tile (with more than one, the
// output must be dense and zero when the GEMM starts adding to it), and the modelled time in us of a call.
struct TriPlan {
    int halves;
    uint32_t ranges;
    double us;
};
TriPlan limb_gemm_tri_plan(uint32_t M, uint32_t NV, uint64_t K, int num_sms);

// out[i * ld_m + v * ld_b] = sum_j D[i][j] X[v][j] mod 2^32 (i < M, v < NV, j < K; one of the strides is 1): a_map covers the
// centred digits (box 64 x 128), b_map the limbs as (K, NV, 3) (box 64 x 32 x 3).
// Launched as the programmatic dependent of the kernel before it in the stream, which makes the limbs (and
// zeroes the output); everything earlier must have completed when that one starts.
cudaError_t launch_limb_gemm_tri(const CUtensorMap &a_map, const CUtensorMap &b_map, const VecSums &sums,
                                 uint32_t *out, uint64_t ld_m, uint64_t ld_b, uint32_t M, uint32_t NV, uint64_t K,
                                 const TriPlan &plan, int num_sms, int *status, cudaStream_t stream);

}  // namespace qpadl

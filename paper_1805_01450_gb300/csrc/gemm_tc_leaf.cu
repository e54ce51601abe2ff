// Tensor-core contractions that multiply a leaf into one operand (gemm_tc.cuh): two steps of the
// program in one pass.
#include "gemm_tc.cuh"

namespace qvx {

cudaError_t launch_gemm_leaf(const GemmArgs &ga, uint32_t nt_cols, cudaStream_t s) {
    return launch_gemm_split<2, true>(ga, nt_cols, s);
}

}  // namespace qvx

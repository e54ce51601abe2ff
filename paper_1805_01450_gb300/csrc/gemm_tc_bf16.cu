// Tensor-core contractions with three-part bf16 operands (gemm_tc.cuh).
#include "gemm_tc.cuh"

namespace qvx {

cudaError_t launch_gemm_bf16(const GemmArgs &ga, uint32_t nt_cols, cudaStream_t s) {
    return launch_gemm_split<3, false>(ga, nt_cols, s);
}

}  // namespace qvx

// Tensor-core contractions: the launch of a step, and the kernels with two-part fp16 operands
// (gemm_tc.cuh).
#include "gemm_tc.cuh"

namespace qvx {

cudaError_t launch_gemm_f16(const GemmArgs &ga, uint32_t nt_cols, cudaStream_t s) {
    return launch_gemm_split<2, false>(ga, nt_cols, s);
}

// real columns of a tile: two per complex column, up to 128 complex columns
uint32_t gemm_nt(const GemmStep &g) { return g.nn >= 7 ? 256u : (2u << g.nn); }

cudaError_t launch_gemm_step(const LaunchArgs &a, const GemmStep &g, const GemmLeaf *leaf, const GemmScale *scale,
                             uint32_t *max_c, int64_t item0, int64_t n_items, float2 *arenas, cudaStream_t s) {
    if (g.nk < 3 || g.nk > 10 || g.nm < 7 || g.nn < 3 || n_items <= 0 || (leaf && !scale))
        return cudaErrorInvalidConfiguration;
    const uint32_t nt_cols = gemm_nt(g);
    GemmArgs ga;
    ga.a = a;
    ga.g = g;
    ga.leaf = leaf ? *leaf : GemmLeaf{};
    ga.sc = scale ? *scale : GemmScale{};
    ga.max_c = max_c;
    ga.item0 = item0;
    ga.n_items = n_items;
    ga.arenas = arenas;
    ga.n_chunks = std::max(1u, (1u << g.nk) / kKq);   // 8 summed entries: one half-filled chunk
    ga.n_mt = (1u << g.nm) / kRows;
    ga.n_nt = (2u << g.nn) / nt_cols;
    ga.mt_bits = (uint32_t)__builtin_ctz(ga.n_mt);
    ga.nt_bits = (uint32_t)__builtin_ctz(ga.n_nt);
    ga.n_tiles = 0;
    ga.run_bits = 0;
    if (leaf) return launch_counted(launch_gemm_leaf(ga, nt_cols, s));
    return launch_counted(scale ? launch_gemm_f16(ga, nt_cols, s) : launch_gemm_bf16(ga, nt_cols, s));
}

}  // namespace qvx

// Dense contractions on the tcgen05 tensor cores (stepwise engine, opts.tensor_cores).
//
// A step C[b, m, n] = sum_k A[b, m, k] B[b, k, n] in complex64 becomes one real GEMM per
// (work item, b): with A = Ar + i Ai and B = Br + i Bi,
//   [Re C[m, n], Im C[m, n]] = [Ar | Ai][m, :]  times  [[Br, Bi], [-Bi, Br]][:, (n, re/im)],
// i.e. the left factor's real summed index is (part p, k) with part 0 = Ar and part 1 = Ai,
// and the right factor has two real columns per complex column n: (Br; -Bi) for Re and
// (Bi; Br) for Im (a tile's Re columns first, then its Im columns). Every real operand x is
// split into 16-bit parts whose products are accumulated in FP32:
//   kParts = 2: x = h + l in fp16 (11 significant bits each, h = rn(x), l = rn(x - h)), three
//     products h*h + h*l + l*h. fp16's range is narrow, so each operand is first multiplied by
//     the power of two that brings its tensor's largest entry (of this work item) to 2^14 ...
//     2^15; the scales are exact and taken out again in the epilogue. Entries down to 2^-16 of
//     the largest keep all 22 bits. The largest entry of a tensor is tracked by the kernel that
//     writes it (note_max).
//   kParts = 3: x = h + m + l in bf16 (8 bits each), the six products h*h + h*m + m*h + h*l +
//     l*h + m*m; the dropped terms are below 2^-23 of the product. It has FP32's range and
//     serves circuits with gates whose own entries differ in size (Plan::fp16_split).
// What limits the accuracy is not the split but the accumulation (group_chunks says how that is
// kept short). Three products instead of six also halve the MMAs and take a third off the operand
// parts stored in and read from shared memory, which bounds the loop. Two bf16 parts with three
// products (about 2^-16 per product) are not accurate enough: on a 64-qubit circuit the
// amplitude moved by 1.2e-5 of its size, above the 1e-5 tolerance.
//
// The row role goes to the operand that holds C's lowest mode, so tensor-memory lane i (row
// m = i of a 128-row tile) holds C entries that are consecutive in memory along the lanes;
// a lane's Re column and Im column n are the two parts of C[m, n], so the epilogue stores
// complex64 values straight from the registers tcgen05.ld fills, coalesced across the warp,
// with no transpose. A tile is 128 complex rows by NT real (NT / 2 complex, up to 128)
// columns of one (item, b). The kernel is persistent (one CTA per SM walks the tiles) and
// warp-specialised: producer warps load the complex64 operands straight from the arena into
// registers (two chunks of 16 summed entries ahead), split them into
// 16-bit parts and store them in the tensor cores' K-major core-matrix layout in a ring
// of shared-memory stages (no separate packing pass: the operands cross HBM once, as
// complex64); one thread issues each chunk's tcgen05.mma (2 parts x 3 or 6 products, K =
// 16 each) into one of two tensor-memory accumulators; epilogue warps store a finished
// accumulator while the next tile's chunks are loaded and multiplied into the other. A step
// with 8 summed entries runs as one chunk whose second half is zeros. Steps whose column tile
// fits in shared memory and that have many row tiles per column tile take the B-stationary form (gemm_tc_bs_kernel,
// below): a column tile's split B stays in shared memory for all the row tiles that use it.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "device_program.h"
#include "device_util.cuh"
#include "kernels.h"

namespace qvx {
namespace {

constexpr uint32_t kRows = 128;        // rows per tile (complex rows of C)
constexpr uint32_t kKq = 16;           // complex summed entries per chunk (one MMA K-step)
constexpr uint32_t kPitch = 272;       // bytes between 8-row groups: two 128-byte core matrices
                                       // along the summed index and 16 bytes that spread the
                                       // producers' 16-byte stores over all banks
constexpr uint32_t kPolls = 1u << 22;
constexpr uint32_t kEpiThreads = 256;  // eight epilogue warps, two per tensor-memory lane quarter

__host__ __device__ constexpr uint32_t region_bytes(uint32_t rows) { return rows / 8u * kPitch; }
// One chunk of B: per bf16 level three consecutive blocks of NT / 2 rows, [-Bi][Br][Bi]. The
// real columns of a tile are all its Re columns, then all its Im columns, so part 0 of the
// right factor is the two blocks [Br][Bi] and part 1 the two blocks [-Bi][Br]: a descriptor
// that starts one block earlier, and Br is stored once. With Re and Im interleaved column by
// column a level took four blocks: with three parts 48 instead of 36 KB of stores per chunk of a
// 256-column tile, whose loop is bound by shared-memory traffic. Together with one barrier arrival
// per warp (warp_arrive) the streaming steps of a 64-qubit circuit, with three parts, went from 2.90
// to 2.56 ms (64 summed entries, 190 -> 215 algorithmic TFLOP/s) and from 1.52 to 1.21 ms (32
// summed, 128 columns).
__host__ __device__ constexpr uint32_t b_block_bytes(uint32_t nt) { return region_bytes(nt / 2u); }
template <int kParts>
__host__ __device__ constexpr uint32_t b_chunk_bytes(uint32_t nt) { return 3u * kParts * b_block_bytes(nt); }
// One stage: A regions (part 0's levels, part 1's levels), then a chunk of B.
template <int kParts>
__host__ __device__ constexpr uint32_t a_bytes() { return 2u * kParts * region_bytes(kRows); }
template <int NT, int kParts>
__host__ __device__ constexpr uint32_t stage_bytes() { return a_bytes<kParts>() + b_chunk_bytes<kParts>(NT); }

// Thread roles, by warpgroup (the unit of setmaxnreg): 256 A producers (one unit of a chunk
// each: 8 summed entries of one of the 128 rows), one B producer per B unit (8 entries of one
// complex column; at least a warpgroup, threads past the units only take part in the barriers),
// a warpgroup whose first warp issues the MMAs, and 256 epilogue threads. A producer holds two
// chunks in registers while a third is split, for which the 72 or 80 registers of an even split
// are too few: the other roles hand registers over.
template <int NT>
__host__ __device__ constexpr uint32_t b_threads() { return NT > 128 ? (uint32_t)NT : 128u; }
template <int NT>
__host__ __device__ constexpr uint32_t mma_warp() { return (256u + b_threads<NT>()) / 32u; }
template <int NT>
__host__ __device__ constexpr uint32_t epi_warp() { return mma_warp<NT>() + 4u; }
template <int NT>
__host__ __device__ constexpr uint32_t block_threads() { return 32u * epi_warp<NT>() + kEpiThreads; }
//
// Registers per thread of a role after the hand-over (streaming form, B-stationary form). The
// shares together stay within those the block is launched with (72 x 896 at 256 columns, 80 x
// 768 below; gemm_grid checks the compiled count before the first launch).
template <int NT>
struct Regs {
    static constexpr uint32_t kLaunch = NT > 128 ? 72u : 80u;
    static constexpr uint32_t kProd = NT > 128 ? 80u : 96u, kIssue = 56u, kEpi = 64u;
    static constexpr uint32_t kBsA = 88u, kBsB = 64u, kBsIssue = 40u, kBsEpi = NT > 128 ? 80u : 96u;
    static_assert((256u + b_threads<NT>()) * kProd + 128u * kIssue + 256u * kEpi <= kLaunch * block_threads<NT>(), "streaming");
    static_assert(256u * kBsA + b_threads<NT>() * kBsB + 128u * kBsIssue + 256u * kBsEpi <= kLaunch * block_threads<NT>(),
                  "B-stationary");
};
template <uint32_t kRegs>
__device__ __forceinline__ void regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegs)); }
template <uint32_t kRegs>
__device__ __forceinline__ void regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegs)); }

// Tensor-memory columns of one accumulator.
template <int NT>
__host__ __device__ constexpr uint32_t acc_cols() { return NT < 32 ? 32u : (uint32_t)NT; }
// Accumulators of the B-stationary form and of sums in runs: the narrower the column tile, the shorter a tile's
// work against its fixed barrier round trips, so narrow tiles keep more tiles in flight
// (tensor memory holds 512 columns: 2 x 256, 4 x 128, 8 x 64, 8 x 32).
template <int NT>
__host__ __device__ constexpr uint32_t bs_accs() { return 512u / acc_cols<NT>() < 8u ? 512u / acc_cols<NT>() : 8u; }
// Operand stages of the shared-memory ring: three, or four for a group of four chunks. With five
// (all that fit at 256 columns) the steps ran 7 to 17 % slower, with two 6 to 8 %: shared memory
// that the ring does not take is L1 cache for the columns.
constexpr uint32_t kStages = 4u;
template <int kParts>
__host__ __device__ constexpr uint32_t n_stages(uint32_t n_chunks) { return kParts == 2 && n_chunks == 4u ? 4u : 3u; }
// complex columns an epilogue warp reads at a time (the same number of Re and Im columns)
template <int NT>
__host__ __device__ constexpr uint32_t epi_cols() { return NT >= 64 ? 16u : 8u; }
template <int NT, int kParts>
__host__ __device__ constexpr size_t smem_bytes(uint32_t stages, uint32_t K) {   // three offset tables (A, B, the leaf)
    return (size_t)stages * stage_bytes<NT, kParts>() + 12u * (size_t)K;
}

__device__ __forceinline__ uint32_t core_offset(uint32_t r, uint32_t g) {
    return (r >> 3) * kPitch + g * 128u + (r & 7u) * 16u;
}

__device__ __forceinline__ const float2 *gemm_operand(const LaunchArgs &a, const float2 *arena, uint64_t ref,
                                                      bool leaf, int64_t item) {
    if (!leaf) return arena + ref;
    const unsigned char *img = a.image;
    const DevProgram *P = reinterpret_cast<const DevProgram *>(img);
    const DevLeaf *leaves = reinterpret_cast<const DevLeaf *>(img + P->leaves_off);
    const float2 *ldata = reinterpret_cast<const float2 *>(img + P->leaf_data_off);
    const Bits x = load_bits(a.bitstrings, item / a.o_count, a.words);
    const uint64_t o = (uint64_t)(a.o_begin + item % a.o_count);
    return ldata + leaf_base(leaves[ref], x, o);
}

// Split of two floats at once into packed pairs (lo in bits 0-15, hi in bits 16-31) of 16-bit
// parts: the first is rn(lo, hi), the next rn of the remainders, and so on; every remainder is
// exact in FP32 and each conversion rounds to nearest even. Two parts: fp16, three: bf16.
__device__ __forceinline__ uint32_t cvt_bf16x2(float lo, float hi) {
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ uint32_t cvt_f16x2(float lo, float hi) {
    uint32_t d;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// x - h for one half of a packed pair (mixed-precision multiply-add: exact, one instruction
// instead of a conversion and a subtraction).
__device__ __forceinline__ void f16x2_rest(uint32_t w, float lo, float hi, float &rl, float &rh) {
    asm("{\n .reg .b16 l, h, m1;\n mov.b32 {l, h}, %2;\n mov.b16 m1, 0xBC00;\n fma.rn.f32.f16 %0, l, m1, %3;\n"
        " fma.rn.f32.f16 %1, h, m1, %4;\n}\n" : "=f"(rl), "=f"(rh) : "r"(w), "f"(lo), "f"(hi));
}
__device__ __forceinline__ float2 scaled2(float2 v, float s) {   // both components in one instruction
    uint64_t r, a, b;
    asm("mov.b64 %0, {%1, %2};" : "=l"(a) : "f"(v.x), "f"(v.y));
    asm("mov.b64 %0, {%1, %1};" : "=l"(b) : "f"(s));
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(r));
    return v;
}

template <int kParts>
__device__ __forceinline__ void split_pair(float lo, float hi, uint32_t (&w)[kParts][4], int p) {
    if constexpr (kParts == 2) {
        const uint32_t H = cvt_f16x2(lo, hi);
        float rl, rh;
        f16x2_rest(H, lo, hi, rl, rh);
        w[0][p] = H;
        w[1][p] = cvt_f16x2(rl, rh);
    } else {
        const uint32_t H = cvt_bf16x2(lo, hi);
        const float rl = lo - bf_lo(H), rh = hi - bf_hi(H);
        const uint32_t M = cvt_bf16x2(rl, rh);
        w[0][p] = H;
        w[1][p] = M;
        w[2][p] = cvt_bf16x2(rl - bf_lo(M), rh - bf_hi(M));
    }
}

// Packed parts (one row per level) of the real and imaginary parts of 8 summed entries of one
// operand row or column: word p holds entries 2p (low) and 2p + 1 (high).
template <int kParts>
__device__ __forceinline__ void split8(const float2 *v, uint32_t (&re)[kParts][4], uint32_t (&im)[kParts][4]) {
#pragma unroll
    for (int p = 0; p < 4; p++) {
        split_pair<kParts>(v[2 * p].x, v[2 * p + 1].x, re, p);
        split_pair<kParts>(v[2 * p].y, v[2 * p + 1].y, im, p);
    }
}

// Power of two that brings a tensor whose largest entry has the bits m (of its absolute value)
// to 2^14 ... 2^15, as a biased float exponent; at most 2^126, and 1 for a tensor that holds an
// infinity or NaN (which then reach the result). Scales are exact; scale_exp returns the
// exponent s of 2^s.
__device__ __forceinline__ uint32_t scale_field(uint32_t m) {
    const uint32_t e = m >> 23;
    return e == 255u ? 127u : min(253u, 268u - e);
}
__device__ __forceinline__ float pow2_field(uint32_t f) { return __uint_as_float(f << 23); }

// What the epilogue multiplies an accumulator by to take out both operands' scales: 2^t with
// t = 254 - fa - fb, in two factors when t is outside the float exponents.
struct Unscale {
    float f1, f2;
    bool two;
};
__device__ __forceinline__ Unscale unscale_of(uint32_t ma, uint32_t mb) {
    const int t = 254 - (int)scale_field(ma) - (int)scale_field(mb);
    const int t1 = max(-126, min(126, t)), t2 = max(-126, min(126, t - t1));
    Unscale u;
    u.f1 = pow2_field((uint32_t)(t1 + 127));
    u.f2 = pow2_field((uint32_t)(t2 + 127));
    u.two = t2 != 0;
    return u;
}
__device__ __forceinline__ float2 unscaled(const Unscale &u, uint32_t re, uint32_t im) {
    float2 c = scaled2(make_float2(__uint_as_float(re), __uint_as_float(im)), u.f1);
    if (u.two) c = scaled2(c, u.f2);
    return c;
}

// Shared-memory matrix descriptor of a K-major tile without swizzling: start address, the
// byte distance between core matrices along the summed index (lbo) and between 8-row groups
// (sbo), descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void mma_f16kind(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
}

// The products of one chunk, 2 parts (Ar, Ai) each: of two fp16 parts the small ones (h*l, l*h)
// and the large one (h*h) apart, of three bf16 parts all six. The accumulator d is overwritten
// by the first product when `first`.
template <int kParts>
struct ChunkDesc {
    uint64_t a[2][kParts], b[2][kParts];
    __device__ __forceinline__ ChunkDesc(uint32_t sa, uint32_t ra, const uint32_t (&sb)[2][kParts]) {
#pragma unroll
        for (uint32_t p = 0; p < 2; p++)
#pragma unroll
            for (uint32_t q = 0; q < (uint32_t)kParts; q++) {
                a[p][q] = smem_desc(sa + (kParts * p + q) * ra, 128u, kPitch);
                b[p][q] = smem_desc(sb[p][q], 128u, kPitch);
            }
    }
};
__device__ __forceinline__ void mma_small(uint32_t d, const ChunkDesc<2> &c, uint32_t idesc, bool first) {
#pragma unroll
    for (uint32_t p = 0; p < 2; p++) {
        mma_f16kind(d, c.a[p][0], c.b[p][1], idesc, !(first && p == 0u));
        mma_f16kind(d, c.a[p][1], c.b[p][0], idesc, 1u);
    }
}
__device__ __forceinline__ void mma_large(uint32_t d, const ChunkDesc<2> &c, uint32_t idesc) {
#pragma unroll
    for (uint32_t p = 0; p < 2; p++) mma_f16kind(d, c.a[p][0], c.b[p][0], idesc, 1u);
}
__device__ __forceinline__ void mma_six(uint32_t d, const ChunkDesc<3> &c, uint32_t idesc, bool first) {
#pragma unroll
    for (uint32_t p = 0; p < 2; p++) {
        mma_f16kind(d, c.a[p][0], c.b[p][0], idesc, !(first && p == 0u));
        mma_f16kind(d, c.a[p][0], c.b[p][1], idesc, 1u);
        mma_f16kind(d, c.a[p][1], c.b[p][0], idesc, 1u);
        mma_f16kind(d, c.a[p][0], c.b[p][2], idesc, 1u);
        mma_f16kind(d, c.a[p][2], c.b[p][0], idesc, 1u);
        mma_f16kind(d, c.a[p][1], c.b[p][1], idesc, 1u);
    }
}

// Instruction descriptor: FP32 accumulator, A and B fp16 (0) or bf16 (1), N = nt, M = 128.
template <int kParts>
__device__ __forceinline__ constexpr uint32_t mma_idesc(uint32_t nt) {
    return (1u << 4) | ((kParts == 3 ? 1u : 0u) << 7) | ((kParts == 3 ? 1u : 0u) << 10) | ((nt >> 3) << 17) | ((kRows >> 4) << 24);
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// The split parts of 8 summed entries of one operand row or column.
template <int kParts>
struct Unit {
    uint32_t re[kParts][4], im[kParts][4];
};

__device__ __forceinline__ uint4 packed(const uint32_t (&w)[4]) { return make_uint4(w[0], w[1], w[2], w[3]); }
__device__ __forceinline__ uint4 negated(const uint32_t (&w)[4]) {
    return make_uint4(w[0] ^ 0x80008000u, w[1] ^ 0x80008000u, w[2] ^ 0x80008000u, w[3] ^ 0x80008000u);
}

// A row m of one summed half (8 entries) in the A regions of a stage (region kParts p +
// level): part 0 takes Ar, part 1 takes Ai.
template <int kParts>
__device__ __forceinline__ void store_a(unsigned char *sa, const Unit<kParts> &x, uint32_t m, uint32_t h) {
    constexpr uint32_t R = region_bytes(kRows);
    const uint32_t o = core_offset(m, h);
#pragma unroll
    for (uint32_t q = 0; q < (uint32_t)kParts; q++) {
        *reinterpret_cast<uint4 *>(sa + q * R + o) = packed(x.re[q]);
        *reinterpret_cast<uint4 *>(sa + (kParts + q) * R + o) = packed(x.im[q]);
    }
}

// Complex B column n of one summed half in the blocks of a chunk (level q: -Bi, Br, Bi).
template <int NT, int kParts>
__device__ __forceinline__ void store_b(unsigned char *sb, const Unit<kParts> &x, uint32_t n, uint32_t h) {
    constexpr uint32_t R = b_block_bytes(NT);
    unsigned char *o = sb + core_offset(n, h);
#pragma unroll
    for (uint32_t q = 0; q < (uint32_t)kParts; q++) {
        *reinterpret_cast<uint4 *>(o + 3u * q * R) = negated(x.im[q]);
        *reinterpret_cast<uint4 *>(o + (3u * q + 1u) * R) = packed(x.re[q]);
        *reinterpret_cast<uint4 *>(o + (3u * q + 2u) * R) = packed(x.im[q]);
    }
}

// The same in regions of NT rows (region kParts p + level): real column 2n takes Br in part 0
// and -Bi in part 1, real column 2n + 1 takes Bi in part 0 and Br in part 1 (the B-stationary
// form: B is stored once per column tile, and its epilogue reads the (Re, Im) column pairs
// with one tensor-memory load; with Re and Im in two halves its largest step took 7.1 instead
// of 6.5 ms).
template <int NT, int kParts>
__device__ __forceinline__ void store_b_interleaved(unsigned char *sb, const Unit<kParts> &x, uint32_t n, uint32_t h) {
    constexpr uint32_t R = region_bytes(NT);
    const uint32_t o0 = core_offset(2u * n, h), o1 = core_offset(2u * n + 1u, h);
#pragma unroll
    for (uint32_t q = 0; q < (uint32_t)kParts; q++) {
        *reinterpret_cast<uint4 *>(sb + q * R + o0) = packed(x.re[q]);
        *reinterpret_cast<uint4 *>(sb + (kParts + q) * R + o0) = negated(x.im[q]);
        *reinterpret_cast<uint4 *>(sb + q * R + o1) = packed(x.im[q]);
        *reinterpret_cast<uint4 *>(sb + (kParts + q) * R + o1) = packed(x.re[q]);
    }
}

// One producer thread's 8 entries of a chunk on their way from memory, and the bits of their
// tensor's largest entry.
struct Fetch {
    float2 v[8];
    uint32_t max;
    uint32_t chunk;                // with a leaf: the chunk, and the leaf's entries for the
    const float2 *factor;          // tile and the thread's row or column
};
template <bool kL2>   // read through L2 only: rows that the SM does not read again
__device__ __forceinline__ void fetch8(Fetch &f, const float2 *src, const uint32_t *off) {
    const uint4 o0 = *reinterpret_cast<const uint4 *>(off), o1 = *reinterpret_cast<const uint4 *>(off + 4);
    const uint32_t o[8] = {o0.x, o0.y, o0.z, o0.w, o1.x, o1.y, o1.z, o1.w};
#pragma unroll
    for (uint32_t j = 0; j < 8; j++) f.v[j] = kL2 ? __ldcg(src + o[j]) : src[o[j]];
}
__device__ __forceinline__ void fetch_zero(Fetch &f) {
#pragma unroll
    for (uint32_t j = 0; j < 8; j++) f.v[j] = make_float2(0.f, 0.f);
    f.max = 0u;
    f.chunk = 0u;
    f.factor = nullptr;
}
template <int kParts>
__device__ __forceinline__ void split_fetch(Fetch &f, Unit<kParts> &x) {
    if constexpr (kParts == 2) {
        const float scale = pow2_field(scale_field(f.max));
#pragma unroll
        for (uint32_t j = 0; j < 8; j++) f.v[j] = scaled2(f.v[j], scale);
    }
    split8<kParts>(f.v, x.re, x.im);
}

// Stage index and phase parity of a ring of S stages, advanced chunk by chunk.
struct RingPos {
    uint32_t s = 0, phase = 0;
    __device__ __forceinline__ void next(uint32_t S) {
        if (++s == S) {
            s = 0;
            phase ^= 1u;
        }
    }
};

// Arrival of a warp whose lanes have each written (and, for operand stages, fenced) their
// share: one per warp; an arrival of every thread serialised hundreds of updates of one
// barrier word per chunk.
__device__ __forceinline__ void warp_arrive(uint32_t bar) {
    __syncwarp();
    if ((threadIdx.x & 31u) == 0u) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// kW accumulator columns of this warp's 32 tensor-memory lanes into registers (one column per
// register). The load and its wait are one asm statement: the registers hold nothing before it.
template <uint32_t kW>
__device__ __forceinline__ void tmem_ld_pairs(uint32_t taddr, uint32_t (&r)[kW]) {
    if constexpr (kW == 32) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
            "%12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, "
            "%30, %31}, [%32];\n tcgen05.wait::ld.sync.aligned;"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
              "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]),
              "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
              "=r"(r[30]), "=r"(r[31])
            : "r"(taddr) : "memory");
    } else if constexpr (kW == 16) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
            "%12, %13, %14, %15}, [%16];\n tcgen05.wait::ld.sync.aligned;"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(taddr) : "memory");
    } else {
        static_assert(kW == 8, "8, 16 or 32 columns");
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                     " tcgen05.wait::ld.sync.aligned;"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                     : "r"(taddr) : "memory");
    }
}
// The same of kW Re columns and kW Im columns, both loads under one wait.
template <uint32_t kW>
__device__ __forceinline__ void tmem_ld(uint32_t re_addr, uint32_t im_addr, uint32_t (&re)[kW], uint32_t (&im)[kW]) {
    if constexpr (kW == 16) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
            "%12, %13, %14, %15}, [%32];\n"
            " tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
            "%28, %29, %30, %31}, [%33];\n tcgen05.wait::ld.sync.aligned;"
            : "=r"(re[0]), "=r"(re[1]), "=r"(re[2]), "=r"(re[3]), "=r"(re[4]), "=r"(re[5]), "=r"(re[6]), "=r"(re[7]),
              "=r"(re[8]), "=r"(re[9]), "=r"(re[10]), "=r"(re[11]), "=r"(re[12]), "=r"(re[13]), "=r"(re[14]), "=r"(re[15]),
              "=r"(im[0]), "=r"(im[1]), "=r"(im[2]), "=r"(im[3]), "=r"(im[4]), "=r"(im[5]), "=r"(im[6]), "=r"(im[7]),
              "=r"(im[8]), "=r"(im[9]), "=r"(im[10]), "=r"(im[11]), "=r"(im[12]), "=r"(im[13]), "=r"(im[14]), "=r"(im[15])
            : "r"(re_addr), "r"(im_addr) : "memory");
    } else {
        static_assert(kW == 8, "8 or 16 columns");
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%16];\n"
                     " tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8, %9, %10, %11, %12, %13, %14, %15}, [%17];\n"
                     " tcgen05.wait::ld.sync.aligned;"
                     : "=r"(re[0]), "=r"(re[1]), "=r"(re[2]), "=r"(re[3]), "=r"(re[4]), "=r"(re[5]), "=r"(re[6]), "=r"(re[7]),
                       "=r"(im[0]), "=r"(im[1]), "=r"(im[2]), "=r"(im[3]), "=r"(im[4]), "=r"(im[5]), "=r"(im[6]), "=r"(im[7])
                     : "r"(re_addr), "r"(im_addr) : "memory");
    }
}

}  // namespace

struct GemmArgs {
    LaunchArgs a;
    GemmStep g;
    GemmLeaf leaf;                 // kernels with a leaf only
    GemmScale sc;                  // the operands' largest entries (fp16 split)
    uint32_t *max_c;               // per item: bits of C's largest entry, or null (not needed)
    int64_t item0, n_items;
    float2 *arenas;
    uint32_t n_chunks, n_mt, n_nt;
    uint32_t stages;               // A stages of the B-stationary form
    uint32_t run_bits;             // log2 of the chunks of an accumulator run (kRuns)
    uint32_t mt_bits, nt_bits;     // log2 of n_mt and n_nt (every tile count is a power of two)
    uint64_t n_tiles;
};
// The launchers of the two splits (fp16: two parts, gemm_tc.cu; bf16: three, gemm_tc_bf16.cu).
cudaError_t launch_gemm_f16(const GemmArgs &ga, uint32_t nt_cols, cudaStream_t s);
cudaError_t launch_gemm_leaf(const GemmArgs &ga, uint32_t nt_cols, cudaStream_t s);   // fp16, with a leaf (gemm_tc_leaf.cu)
cudaError_t launch_gemm_bf16(const GemmArgs &ga, uint32_t nt_cols, cudaStream_t s);

namespace {

// Bits of an operand's largest entry for item il of the launch; with the leaf multiplied in, of
// a bound on it (a component of a product is at most twice the product of the components).
__device__ __forceinline__ uint32_t operand_max(const uint32_t *max, uint32_t leaf_max, int64_t il) {
    return max ? __ldg(max + il) : leaf_max;
}
template <bool kLeaf>
__device__ __forceinline__ uint32_t side_max(const GemmArgs &ga, bool rows, int64_t il) {
    uint32_t m = rows ? operand_max(ga.sc.max_a, ga.sc.leaf_max_a, il) : operand_max(ga.sc.max_b, ga.sc.leaf_max_b, il);
    if (kLeaf && rows == (ga.leaf.on_rows != 0))
        m = __float_as_uint(2.f * __uint_as_float(m) * __uint_as_float(ga.sc.leaf_max_d)) & 0x7fffffffu;
    return m;
}

// The leaf's entries for one item; the caller adds the offsets of b and of the row or column.
__device__ __forceinline__ const float2 *leaf_entries(const GemmArgs &ga, int64_t item) {
    return gemm_operand(ga.a, nullptr, ga.leaf.leaf, true, item);
}
// 8 summed entries of an operand times the leaf's (off: their offsets in the leaf).
__device__ __forceinline__ void times_leaf(Fetch &f, const float2 *d, const uint32_t *off) {
    const uint4 o0 = *reinterpret_cast<const uint4 *>(off), o1 = *reinterpret_cast<const uint4 *>(off + 4);
    const uint32_t o[8] = {o0.x, o0.y, o0.z, o0.w, o1.x, o1.y, o1.z, o1.w};
#pragma unroll
    for (uint32_t j = 0; j < 8; j++) {
        const float2 y = __ldg(d + o[j]), x = f.v[j];
        f.v[j] = make_float2(x.x * y.x - x.y * y.y, x.x * y.y + x.y * y.x);
    }
}

// Bounded mbarrier wait that also gives up once another role has set the CTA's fail flag.
__device__ __forceinline__ bool wait_or_fail(uint32_t bar, uint32_t parity, volatile int *fail) {
    for (uint32_t i = 0; i < kPolls; i++) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((i & 63u) == 63u && *fail) return false;
    }
    return false;
}

// The same for a whole warp, with one answer for all its lanes: the roles' loops contain
// warp-wide operations, so their lanes must leave them together.
__device__ __forceinline__ bool warp_wait_or_fail(uint32_t bar, uint32_t parity, volatile int *fail) {
    return __all_sync(0xffffffffu, wait_or_fail(bar, parity, fail));
}

// The tensor cores truncate the accumulator at every MMA, relative to the value that it has by
// then, so a long sum comes out too small (by 3e-8 a truncation in the mean, over three times the
// rounding of an FP32 sum of such length). Two parts of fp16 keep the truncations of full size few:
//  - chunks go to an accumulator in groups of two or four, first the small products (h*l, l*h) of
//    all of them, then the large ones: an MMA costs accuracy only once large products are in, 2 of
//    a chunk's 6 instead of all;
//  - sums of more chunks run in several accumulators, added in FP32 by the epilogue (kRuns):
//    a tile has a pair of them, the first for its first run and the sum, the second for the others.
// Slice terms of 64-qubit circuits, relative error against FP64: 5.9e-7, 6.5e-7 and 9.4e-7
// (all products in order in one accumulator: 6e-6, 2.9e-6 and 5.4e-6 too small; six bf16 products,
// without merged steps: 3.3e-6, 2.3e-6 and 4.2e-6), and sums that need no rounding are exact.
// A constant gain in place of this is right for no particular sum.
template <int kParts>
__host__ __device__ constexpr uint32_t group_chunks() { return kParts == 2 ? 2u : 1u; }

// Accumulator of run r of the CTA's tile number n, and how often it was used before.
template <uint32_t NA>
struct RunSlot {
    uint32_t buf, uses;
    __device__ __forceinline__ RunSlot(uint32_t n, uint32_t r, uint32_t runs) {
        const uint32_t before = n / (NA / 2u);
        buf = 2u * (n % (NA / 2u)) + (r ? 1u : 0u);
        uses = r ? before * (runs - 1u) + r - 1u : before;
    }
};

// The MMA thread's part of a group of n chunks, from the ring's next stages into accumulator d:
// waits for the stages, issues the products, and commits the stages' release. first: the group
// overwrites the accumulator. b_at(i, s, bs): the addresses of the B parts of the group's chunk i
// (ring stage s) into bs.
template <int kParts, class BAt>
__device__ __forceinline__ bool mma_group(uint32_t d, uint32_t n, bool first, RingPos &ring, uint32_t S, uint32_t stages,
                                          uint32_t stage_bytes, uint32_t region, uint64_t *full, uint64_t *empty, const BAt &b_at,
                                          uint32_t idesc, volatile int *fail) {
    RingPos at = ring;
    for (uint32_t i = 0; i < n; i++, at.next(S)) {
        if (!wait_or_fail(smem_u32(&full[at.s]), at.phase, fail)) return false;
        tc_fence_after();
        uint32_t bs[2][kParts];
        b_at(i, at.s, bs);
        const ChunkDesc<kParts> c(stages + at.s * stage_bytes, region, bs);
        if constexpr (kParts == 2) mma_small(d, c, idesc, first && i == 0u);
        else mma_six(d, c, idesc, first && i == 0u);
    }
    if constexpr (kParts == 2) {
        at = ring;
        for (uint32_t i = 0; i < n; i++, at.next(S)) {
            uint32_t bs[2][kParts];
            b_at(i, at.s, bs);
            mma_large(d, ChunkDesc<kParts>(stages + at.s * stage_bytes, region, bs), idesc);
            mma_commit(smem_u32(&empty[at.s]));
        }
    } else {
        mma_commit(smem_u32(&empty[ring.s]));
    }
    ring = at;
    return true;
}

// Adds kW accumulator columns to registers, and to other columns (tensor memory), in FP32.
template <uint32_t kW>
__device__ __forceinline__ void add_columns(uint32_t (&sum)[kW], uint32_t taddr) {
    uint32_t v[kW];
    tmem_ld_pairs<kW>(taddr, v);
#pragma unroll
    for (uint32_t i = 0; i < kW; i++) sum[i] = __float_as_uint(__uint_as_float(sum[i]) + __uint_as_float(v[i]));
}
template <uint32_t kW>
__device__ __forceinline__ void tmem_add(uint32_t to, uint32_t from) {
    uint32_t v[kW];
    tmem_ld_pairs<kW>(to, v);
    add_columns<kW>(v, from);
    if constexpr (kW == 16) {
        asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                     "%13, %14, %15, %16};\n tcgen05.wait::st.sync.aligned;" ::"r"(to),
                     "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
                     "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
                     : "memory");
    } else {
        static_assert(kW == 8, "8 or 16 columns");
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n"
                     " tcgen05.wait::st.sync.aligned;" ::"r"(to),
                     "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                     : "memory");
    }
}

struct TileCoord {
    uint32_t mt, nt, beta;
    int64_t il;
};

// Tile t's row tile, column tile, batch index and work item: row tiles of one (item, b) and
// column tile run next to each other. All counts are powers of two, so shifts and masks.
__device__ __forceinline__ TileCoord tile_coord(uint64_t t, const GemmArgs &ga) {
    TileCoord c;
    c.mt = (uint32_t)t & (ga.n_mt - 1u);
    t >>= ga.mt_bits;
    c.nt = (uint32_t)t & (ga.n_nt - 1u);
    t >>= ga.nt_bits;
    c.il = (int64_t)(t >> ga.g.nb);
    c.beta = (uint32_t)t & ((1u << ga.g.nb) - 1u);
    return c;
}

// Tile order of the B-stationary form: row tiles fastest (one column tile's B serves a run of
// them), then batch index and work item, column tile slowest. The CTAs' contiguous ranges
// then walk the column tiles of one (item, b) at the same time on different SMs, so the
// second column tile's A rows are still in L2 (with the column tile next to the row tiles,
// one CTA read each A tile twice, some 32 row tiles apart, from HBM).
__device__ __forceinline__ TileCoord tile_coord_bs(uint64_t t, const GemmArgs &ga) {
    TileCoord c;
    c.mt = (uint32_t)t & (ga.n_mt - 1u);
    t >>= ga.mt_bits;
    c.beta = (uint32_t)t & ((1u << ga.g.nb) - 1u);
    t >>= ga.g.nb;   // below n_items * n_nt < 2^32: a 32-bit division (a 64-bit one is a
                     // called routine, and the kernel's loops lost a tenth to it)
    const uint32_t q = (uint32_t)t, n = (uint32_t)ga.n_items;
    c.il = (int64_t)(q % n);
    c.nt = q / n;
    return c;
}

// The coordinates of consecutive tiles in that order, advanced without a division (the item
// count need not be a power of two).
struct BsCursor {
    TileCoord c;
    __device__ __forceinline__ void next(const GemmArgs &ga) {
        if (++c.mt < ga.n_mt) return;
        c.mt = 0;
        if (++c.beta < (1u << ga.g.nb)) return;
        c.beta = 0;
        if (++c.il < ga.n_items) return;
        c.il = 0;
        c.nt++;
    }
    // the first row tile of the next column tile
    __device__ __forceinline__ void next_group(const GemmArgs &ga) {
        c.mt = ga.n_mt - 1u;
        next(ga);
    }
};

// Persistent, warp-specialised tensor-core contraction. One CTA per SM walks the tiles
// t = blockIdx.x, blockIdx.x + gridDim.x, ... (128 rows x NT real columns of one (item, b)):
//   producer warps (one operand unit per thread): load the unit's 8 complex64 entries of a
//              chunk into registers, two chunks ahead and across tile boundaries, scale and
//              split them, store the parts into the next stage of the ring and arrive on the
//              stage's "full" barrier. (Through private shared-memory slots filled by cp.async,
//              two to four chunks ahead, the copies and their reads were half of the
//              shared-memory traffic: s134 of circuit 5003, 128 summed entries, 2.52 ms, 2.11
//              with registers.)
//   one warp   allocates two tensor-memory accumulators; one thread issues each chunk's
//              tcgen05.mma into the tile's accumulator (the tile's first product
//              overwrites it), commits each chunk to the stage's "empty" barrier and the
//              tile's last chunk to the accumulator's "full" barrier;
//   8 warps    epilogue: wait for an accumulator, read it with tcgen05.ld (warp w reads
//              tensor-memory lanes 32 (w mod 4) ..., i.e. rows 32 (w mod 4) + lane; the two
//              warps of a lane quarter take alternate blocks of complex columns), store each
//              (Re, Im) column pair as one complex64 entry of C and release the accumulator.
//              Four warps left the epilogue about a tenth slower on output-heavy steps: each
//              waits out its tensor-memory reads block by block.
// With two accumulators the epilogue of one tile overlaps the loads and MMAs of the next.
// Every wait is bounded; a wait that runs out sets the CTA's fail flag, the other roles
// leave their loops, the MMA thread waits (bounded) for its issued MMAs before the tensor
// memory is freed, and QVX_ETIMEOUT goes to the status word.
// kLeaf: one operand is multiplied by a leaf between its load and its split, so that a
// contraction and the leaf contraction of its result are one pass with a longer summed index
// (find_pairs in planner.cpp). kRuns: a tile's sum in several accumulator runs.
template <int NT, int kParts, bool kLeaf, bool kRuns>
__global__ void __launch_bounds__(block_threads<NT>(), 1) gemm_tc_kernel(GemmArgs ga) {
    constexpr uint32_t kMmaWarp = mma_warp<NT>(), kEpiWarp = epi_warp<NT>();
    const uint32_t S = n_stages<kParts>(ga.n_chunks);
    constexpr uint32_t kCols = acc_cols<NT>(), NA = kRuns ? bs_accs<NT>() : 2u;   // accumulators
    constexpr uint32_t kRegA = region_bytes(kRows), kStage = stage_bytes<NT, kParts>();
    constexpr uint32_t kW = epi_cols<NT>();
    constexpr uint32_t kNc = (uint32_t)NT / 2u;   // complex columns per tile
    extern __shared__ __align__(1024) unsigned char gsm[];
    __shared__ __align__(8) uint64_t full_bar[kStages], empty_bar[kStages], accf_bar[NA], acce_bar[NA], drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int fail;
    const GemmStep &g = ga.g;
    const uint32_t warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t sbase = smem_u32(gsm);
    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < S; s++) {
            mbar_init(smem_u32(&full_bar[s]), kMmaWarp);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        for (uint32_t b = 0; b < NA; b++) {
            mbar_init(smem_u32(&accf_bar[b]), 1);
            mbar_init(smem_u32(&acce_bar[b]), kEpiThreads / 32u);
        }
        mbar_init(smem_u32(&drain_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fail = 0;
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(NA * kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // the summed index's offsets in A and B (bit-run maps evaluated once per CTA)
    const uint32_t K = ga.n_chunks * kKq;
    uint32_t *tka = reinterpret_cast<uint32_t *>(gsm + S * kStage);
    uint32_t *tkb = tka + K, *tkd = tkb + K;
    for (uint32_t i = threadIdx.x; i < K; i += block_threads<NT>()) {
        tka[i] = pext_runs(i, g.ak, g.n_ak);
        tkb[i] = pext_runs(i, g.bk, g.n_bk);
        if (kLeaf) tkd[i] = pext_runs(i, ga.leaf.k, ga.leaf.n_k);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    if (warp < kMmaWarp) {
        regs_inc<Regs<NT>::kProd>();
        // producer: unit u < 256 is A row m = mt*128 + (u & 127), summed half u >> 7; unit
        // u >= 256 is complex B column n = nt*NT/2 + (u - 256) % (NT/2), summed half
        // (u - 256) / (NT/2)
        const uint32_t u = threadIdx.x;
        const bool is_a = u < 256u;
        const bool active = is_a || u - 256u < (uint32_t)NT;
        const uint32_t row = is_a ? (u & 127u) : (u - 256u) % kNc;
        const uint32_t h = is_a ? (u >> 7) : ((u - 256u) / kNc) & 1u;
        const uint32_t *koff = (is_a ? tka : tkb) + 8u * h;
        // a step with 8 summed entries fills one chunk's first half: the units of the second
        // half load nothing and store zeros, which add nothing to the products
        const bool loads = active && !((1u << g.nk) < kKq && h == 1u);
        // the part of the operand's offset that is the thread's own; the tile's part is the
        // same for the whole block
        const uint32_t own = is_a ? pext_runs(row, g.am, g.n_am) : pext_runs(row, g.bn, g.n_bn);
        const bool scaled = kLeaf && loads && is_a == (ga.leaf.on_rows != 0);   // the leaf's side
        const uint32_t own_d = kLeaf ? pext_runs(row, ga.leaf.r, ga.leaf.n_r) : 0u;
        // load cursor: the tile and chunk that are loaded next
        uint64_t lt = blockIdx.x;
        uint32_t lc = 0, tile_max = 0;
        const float2 *src = nullptr, *factor = nullptr;
        auto setup = [&]() {
            const TileCoord tc = tile_coord(lt, ga);
            const float2 *arena = ga.arenas + (uint64_t)tc.il * ga.a.arena_elems;
            const uint32_t ta = pext_runs(tc.beta, g.ab, g.n_ab) + pext_runs(tc.mt * kRows, g.am, g.n_am);
            const uint32_t tb = pext_runs(tc.beta, g.bb, g.n_bb) + pext_runs(tc.nt * kNc, g.bn, g.n_bn);
            src = (is_a ? gemm_operand(ga.a, arena, g.a_off, g.flags & kStepALeaf, ga.item0 + tc.il) + ta
                        : gemm_operand(ga.a, arena, g.b_off, g.flags & kStepBLeaf, ga.item0 + tc.il) + tb) + own;
            if (kParts == 2) tile_max = side_max<kLeaf>(ga, is_a, tc.il);
            if (kLeaf && scaled)
                factor = leaf_entries(ga, ga.item0 + tc.il) + pext_runs(tc.beta, ga.leaf.b, ga.leaf.n_b) + own_d +
                         pext_runs(is_a ? tc.mt * kRows : tc.nt * kNc, ga.leaf.r, ga.leaf.n_r);
        };
        auto fetch = [&](Fetch &f) {
            if (lt >= ga.n_tiles) return;
            if (loads) fetch8<true>(f, src, koff + lc * kKq);
            if (kLeaf) {
                f.factor = factor;
                f.chunk = lc;
            }
            f.max = tile_max;
            if (++lc == ga.n_chunks) {
                lc = 0;
                lt += gridDim.x;
                if (lt < ga.n_tiles) setup();
            }
        };
        setup();
        const uint64_t my_tiles = (ga.n_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x;
        const uint64_t total = my_tiles * ga.n_chunks;
        RingPos ring;
        // splits a loaded chunk, starts the load of the one after next into the same registers,
        // and stores the parts once the stage is free
        auto produce = [&](Fetch &f) -> bool {
            Unit<kParts> x;
            if (kLeaf && scaled) times_leaf(f, f.factor, tkd + f.chunk * kKq + 8u * h);
            split_fetch<kParts>(f, x);
            fetch(f);
            if (!warp_wait_or_fail(smem_u32(&empty_bar[ring.s]), ring.phase ^ 1u, &fail)) {
                fail = 1;
                return false;
            }
            unsigned char *sa = gsm + ring.s * kStage;
            if (is_a) store_a<kParts>(sa, x, row, h);
            else if (active) store_b<NT, kParts>(sa + a_bytes<kParts>(), x, row, h);
            // the generic-proxy stores must be visible to the tensor cores' reads
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            warp_arrive(smem_u32(&full_bar[ring.s]));
            ring.next(S);
            return true;
        };
        Fetch f0, f1;
        fetch_zero(f0);
        fetch_zero(f1);
        fetch(f0);
        fetch(f1);
        for (uint64_t gc = 0; gc < total; gc += 2) {
            if (!produce(f0)) break;
            if (gc + 1 < total && !produce(f1)) break;
        }
    } else if (warp < kEpiWarp) {
        regs_dec<Regs<NT>::kIssue>();
        if (warp == kMmaWarp && lane == 0) {   // MMA issuer
            constexpr uint32_t idesc = mma_idesc<kParts>(NT);
            constexpr uint32_t kBlkB = b_block_bytes(NT);
            const uint32_t group = min(kParts == 2 && !kRuns ? 4u : group_chunks<kParts>(), ga.n_chunks), runs = ga.n_chunks >> ga.run_bits;
            RingPos ring;
            uint32_t j = 0;
            bool ok = true;
            auto b_at = [&](uint32_t, uint32_t stage, uint32_t (&bs)[2][kParts]) {
                const uint32_t sb = sbase + stage * kStage + a_bytes<kParts>();
#pragma unroll
                for (uint32_t q = 0; q < (uint32_t)kParts; q++) {
                    bs[0][q] = sb + (3u * q + 1u) * kBlkB;   // [Br][Bi]
                    bs[1][q] = sb + 3u * q * kBlkB;          // [-Bi][Br]
                }
            };
            for (uint64_t t = blockIdx.x; t < ga.n_tiles && ok; t += gridDim.x, j++) {
                for (uint32_t c = 0; c < ga.n_chunks && ok; c += group) {
                    const uint32_t run = c >> ga.run_bits, at = kRuns ? c & ((1u << ga.run_bits) - 1u) : c;
                    const RunSlot<NA> slot(j, run, runs);
                    const bool starts = at == 0u, ends = kRuns ? run != 0u && at + group == 1u << ga.run_bits : c + group >= ga.n_chunks;
                    const uint32_t buf = kRuns ? slot.buf : j % NA;
                    if (starts) {
                        ok = wait_or_fail(smem_u32(&acce_bar[buf]), ((kRuns ? slot.uses : j / NA) & 1u) ^ 1u, &fail);
                        if (!ok) break;
                        tc_fence_after();
                    }
                    ok = mma_group<kParts>(tmem + buf * kCols, group, starts, ring, S, sbase, kStage, kRegA, full_bar, empty_bar, b_at,
                                           idesc, &fail);
                    if (ok && ends) mma_commit(smem_u32(&accf_bar[buf]));
                }
            }
            if (!ok) fail = 1;
            // every MMA issued so far completes before the tensor memory is freed
            mma_commit(smem_u32(&drain_bar));
            if (!mbar_wait(smem_u32(&drain_bar), 0, kPolls)) fail = 1;
        }
        __syncwarp();
    } else {
        regs_dec<Regs<NT>::kEpi>();
        // epilogue: warp w reads tensor-memory lanes 32q ... 32q + 31 (q = w mod 4): row
        // m = mt*128 + 32q + lane of the tile, whose columns j and NT/2 + j are Re and Im of
        // C[m, nt*NT/2 + j]. For each column the warp's 32 stores are 32 rows, consecutive
        // in C when its lowest modes are row modes (the planner gives the row role to the
        // operand that holds C's lowest mode).
        const uint32_t q = warp & 3u;
        const uint32_t share = (warp - kEpiWarp) >> 2;   // the two warps of a lane quarter split its columns
        uint32_t j = 0;
        bool ok = true;
        // this lane's row of C in a tile
        auto row_of = [&](const TileCoord &tc) {
            return ga.arenas + (uint64_t)tc.il * ga.a.arena_elems + g.c_off + pext_runs(tc.beta, g.cb, g.n_cb) +
                   pext_runs(tc.mt * kRows + 32u * q + lane, g.cm, g.n_cm);
        };
        uint32_t coff[kW];   // offsets of a block's columns in C
#pragma unroll
        for (uint32_t i = 0; i < kW; i++) coff[i] = pext_runs(i, g.cn, g.n_cn);
        const uint32_t lanes = tmem + ((q * 32u) << 16);
        const uint32_t runs = ga.n_chunks >> ga.run_bits;
        for (uint64_t t = blockIdx.x; t < ga.n_tiles; t += gridDim.x, j++) {
            const TileCoord tc = tile_coord(t, ga);
            const RunSlot<NA> last(j, runs - 1u, runs);   // the last run, added to the sum as it is stored
            const uint32_t buf = kRuns ? last.buf : j % NA;
            float2 *Crow = row_of(tc);   // while the MMAs run
            Unscale un{1.f, 1.f, false};
            if (kParts == 2) un = unscale_of(side_max<kLeaf>(ga, true, tc.il), side_max<kLeaf>(ga, false, tc.il));
            uint32_t largest = 0;
            if constexpr (kRuns) {
                for (uint32_t r = 1; r + 1u < runs && ok; r++) {
                    ok = warp_wait_or_fail(smem_u32(&accf_bar[buf]), RunSlot<NA>(j, r, runs).uses & 1u, &fail);
                    if (!ok) break;
                    tc_fence_after();
                    for (uint32_t j0 = share * kW; j0 < (uint32_t)NT; j0 += 2u * kW)
                        tmem_add<kW>(lanes + (buf - 1u) * kCols + j0, lanes + buf * kCols + j0);
                    tc_fence_before();
                    warp_arrive(smem_u32(&acce_bar[buf]));
                }
            }
            if (ok) ok = warp_wait_or_fail(smem_u32(&accf_bar[buf]), (kRuns ? last.uses : j / NA) & 1u, &fail);
            if (!ok) break;
            tc_fence_after();
            const uint32_t taddr = lanes + buf * kCols;
            for (uint32_t j0 = share * kW; j0 < kNc; j0 += 2u * kW) {
                float2 *Cblk = Crow + pext_runs(tc.nt * kNc + j0, g.cn, g.n_cn);
                uint32_t re[kW], im[kW];
                tmem_ld<kW>(taddr + j0, taddr + kNc + j0, re, im);
                if constexpr (kRuns) {
                    add_columns<kW>(re, taddr - kCols + j0);
                    add_columns<kW>(im, taddr - kCols + kNc + j0);
                }
#pragma unroll
                for (uint32_t i = 0; i < kW; i++) {
                    const float2 c = kParts == 2 ? unscaled(un, re[i], im[i])
                                                 : make_float2(__uint_as_float(re[i]), __uint_as_float(im[i]));
                    Cblk[coff[i]] = c;
                    if (ga.max_c) largest = abs_max(largest, c);
                }
            }
            // the accumulator's reads are done: the MMAs of a later tile may reuse it
            tc_fence_before();
            warp_arrive(smem_u32(&acce_bar[buf]));
            if (kRuns) warp_arrive(smem_u32(&acce_bar[buf - 1u]));
            if (ga.max_c) note_max_warp(ga.max_c + tc.il, largest);
        }
        if (!ok) fail = 1;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(NA * kCols) : "memory");
    }
    if (fail && threadIdx.x == 0) atomicCAS(ga.a.status, 0u, 4u /* QVX_ETIMEOUT */);
}

// B-stationary form for steps whose column tile fits in shared memory with all its chunks (64
// summed entries at 256 real columns, twice as many per halving of the columns) and many
// row tiles per column tile: a CTA walks a contiguous range of tiles, row tiles fastest, so
// one column tile's B operand (all its chunks) is split once into resident shared-memory
// regions and serves every row tile of the range that shares it; only A goes through the
// stage ring. The B producers reload when the column tile changes, after the MMAs that read
// the old one have completed. Against the streaming form this removes B's loads, splits and
// stores from the loop (64-qubit circuit 5001: s118, 64 summed entries, 2.56 -> 1.88 ms, 292
// algorithmic TFLOP/s).
template <int NT, int kParts>
__host__ __device__ constexpr uint32_t bs_b_bytes() { return 2u * kParts * region_bytes(NT); }   // one chunk of B
// real accumulator columns an epilogue warp reads at a time
template <int NT>
__host__ __device__ constexpr uint32_t bs_epi_cols() { return NT < 32 ? (uint32_t)NT : 32u; }
// Most chunks of a column tile's B that stay resident, and the A stages beside them (three at
// least, eight at most).
constexpr uint32_t kBsStages = 8u;
constexpr uint32_t kBsBytes = 222u << 10;
template <int NT, int kParts>
__host__ __device__ constexpr uint32_t bs_chunks() {
    uint32_t c = 2u;
    while (2u * c * kKq <= 1024u && 2u * c * bs_b_bytes<NT, kParts>() + 3u * a_bytes<kParts>() + 12u * 2u * c * kKq <= kBsBytes) c *= 2u;
    return c;
}
template <int NT, int kParts>
constexpr uint32_t bs_stages(uint32_t n_chunks) {
    const uint32_t fit = (kBsBytes - n_chunks * (bs_b_bytes<NT, kParts>() + 12u * kKq)) / a_bytes<kParts>();
    return fit < kBsStages ? fit : kBsStages;
}

template <int NT, int kParts, bool kLeaf, bool kRuns>   // as gemm_tc_kernel
__global__ void __launch_bounds__(block_threads<NT>(), 1) gemm_tc_bs_kernel(GemmArgs ga) {
    const uint32_t S = ga.stages;
    constexpr uint32_t NA = bs_accs<NT>();
    constexpr uint32_t PA = 256u, PB = b_threads<NT>();
    constexpr uint32_t kMmaWarp = mma_warp<NT>(), kEpiWarp = epi_warp<NT>();
    constexpr uint32_t kCols = acc_cols<NT>();
    constexpr uint32_t kRegA = region_bytes(kRows), kRegB = region_bytes(NT);
    constexpr uint32_t kStage = a_bytes<kParts>(), kBChunk = bs_b_bytes<NT, kParts>();
    constexpr uint32_t kW = bs_epi_cols<NT>();
    constexpr uint32_t kNc = (uint32_t)NT / 2u;
    extern __shared__ __align__(1024) unsigned char gsm[];
    __shared__ __align__(8) uint64_t full_bar[kBsStages], empty_bar[kBsStages], accf_bar[NA], acce_bar[NA], bfull_bar, bempty_bar, drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int fail;
    const GemmStep &g = ga.g;
    const uint32_t warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t sbase = smem_u32(gsm);
    unsigned char *sB = gsm + S * kStage;                          // resident B, one region set per chunk
    const uint32_t K = ga.n_chunks * kKq;
    uint32_t *tka = reinterpret_cast<uint32_t *>(sB + ga.n_chunks * kBChunk);
    uint32_t *tkb = tka + K, *tkd = tkb + K;
    // this CTA's contiguous range of tiles
    const uint64_t t0 = (uint64_t)blockIdx.x * ga.n_tiles / gridDim.x;
    const uint64_t t1 = ((uint64_t)blockIdx.x + 1u) * ga.n_tiles / gridDim.x;
    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < S; s++) {
            mbar_init(smem_u32(&full_bar[s]), PA / 32u);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        for (uint32_t b = 0; b < NA; b++) {
            mbar_init(smem_u32(&accf_bar[b]), 1);
            mbar_init(smem_u32(&acce_bar[b]), kEpiThreads / 32u);
        }
        mbar_init(smem_u32(&bfull_bar), PB / 32u);
        mbar_init(smem_u32(&bempty_bar), 1);
        mbar_init(smem_u32(&drain_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fail = 0;
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(NA * kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (uint32_t i = threadIdx.x; i < K; i += block_threads<NT>()) {
        tka[i] = pext_runs(i, g.ak, g.n_ak);
        tkb[i] = pext_runs(i, g.bk, g.n_bk);
        if (kLeaf) tkd[i] = pext_runs(i, ga.leaf.k, ga.leaf.n_k);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const bool k8 = (1u << g.nk) < kKq;   // 8 summed entries: the second half of the chunk is zero
    if (warp < PA / 32u) {
        regs_inc<Regs<NT>::kBsA>();
        // A producers: unit u is row u & 127 of the tile, summed half u >> 7
        const uint32_t u = threadIdx.x;
        const uint32_t row = u & 127u, h = u >> 7;
        const bool pad = k8 && h == 1u;
        const uint32_t *koff = tka + 8u * h;
        uint64_t lt = t0;
        uint32_t lc = 0;
        const float2 *src = nullptr, *factor = nullptr;
        uint32_t tile_max = 0;
        const bool scaled = kLeaf && !pad && ga.leaf.on_rows != 0;   // the leaf goes with the rows
        const uint32_t own_d = kLeaf && scaled ? pext_runs(row, ga.leaf.r, ga.leaf.n_r) : 0u;
        BsCursor cur;
        cur.c = tile_coord_bs(t0, ga);
        const uint32_t own = pext_runs(row, g.am, g.n_am);
        auto setup = [&]() {
            const TileCoord &tc = cur.c;
            const float2 *arena = ga.arenas + (uint64_t)tc.il * ga.a.arena_elems;
            if (kParts == 2) tile_max = side_max<kLeaf>(ga, true, tc.il);
            if (kLeaf && scaled)
                factor = leaf_entries(ga, ga.item0 + tc.il) + pext_runs(tc.beta, ga.leaf.b, ga.leaf.n_b) + own_d +
                         pext_runs(tc.mt * kRows, ga.leaf.r, ga.leaf.n_r);
            src = gemm_operand(ga.a, arena, g.a_off, g.flags & kStepALeaf, ga.item0 + tc.il) +
                  pext_runs(tc.beta, g.ab, g.n_ab) + pext_runs(tc.mt * kRows, g.am, g.n_am) + own;
        };
        auto fetch = [&](Fetch &f) {
            if (lt >= t1) return;
            if (!pad) fetch8<false>(f, src, koff + lc * kKq);
            if (kLeaf) {
                f.factor = factor;
                f.chunk = lc;
            }
            f.max = tile_max;
            if (++lc == ga.n_chunks) {
                lc = 0;
                if (++lt < t1) {
                    cur.next(ga);
                    setup();
                }
            }
        };
        if (t0 < t1) setup();
        const uint64_t total = (t1 - t0) * ga.n_chunks;
        RingPos ring;
        auto produce = [&](Fetch &f) -> bool {   // as in the streaming form
            Unit<kParts> x;
            if (kLeaf && scaled) times_leaf(f, f.factor, tkd + f.chunk * kKq + 8u * h);
            split_fetch<kParts>(f, x);
            fetch(f);
            if (!warp_wait_or_fail(smem_u32(&empty_bar[ring.s]), ring.phase ^ 1u, &fail)) {
                fail = 1;
                return false;
            }
            store_a<kParts>(gsm + ring.s * kStage, x, row, h);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            warp_arrive(smem_u32(&full_bar[ring.s]));
            ring.next(S);
            return true;
        };
        Fetch f0, f1;
        fetch_zero(f0);
        fetch_zero(f1);
        fetch(f0);
        fetch(f1);
        for (uint64_t gc = 0; gc < total; gc += 2) {
            if (!produce(f0)) break;
            if (gc + 1 < total && !produce(f1)) break;
        }
    } else if (warp < kMmaWarp) {
        regs_dec<Regs<NT>::kBsB>();
        // B producers: unit v is complex column v % (NT/2) of the column tile, summed half
        // (v / (NT/2)) & 1; once per column tile of the range, every chunk into its region
        const uint32_t v = threadIdx.x - PA;
        const bool active = v < (uint32_t)NT;
        const uint32_t col = v % kNc, h = (v / kNc) & 1u;
        const bool pad = k8 && h == 1u;
        const uint32_t *koff = tkb + 8u * h;
        const bool loads = active && !pad;
        uint32_t gi = 0;
        BsCursor cur;
        cur.c = tile_coord_bs(t0, ga);
        Fetch f;
        fetch_zero(f);
        for (uint64_t t = t0; t < t1; gi++) {
            const uint64_t grp = t >> ga.mt_bits;
            const TileCoord &tc = cur.c;
            const float2 *arena = ga.arenas + (uint64_t)tc.il * ga.a.arena_elems;
            const float2 *src = gemm_operand(ga.a, arena, g.b_off, g.flags & kStepBLeaf, ga.item0 + tc.il) +
                                pext_runs(tc.beta, g.bb, g.n_bb) + pext_runs(tc.nt * kNc + (active ? col : 0u), g.bn, g.n_bn);
            // the first chunk is loaded while the old column tile's last MMAs run
            if (loads) fetch8<false>(f, src, koff);
            f.max = side_max<kLeaf>(ga, false, tc.il);
            const float2 *factor = nullptr;
            const bool scaled = kLeaf && loads && ga.leaf.on_rows == 0;   // the leaf goes with the columns
            if (scaled)
                factor = leaf_entries(ga, ga.item0 + tc.il) + pext_runs(tc.beta, ga.leaf.b, ga.leaf.n_b) +
                         pext_runs(tc.nt * kNc + (active ? col : 0u), ga.leaf.r, ga.leaf.n_r);
            if (!warp_wait_or_fail(smem_u32(&bempty_bar), (gi & 1u) ^ 1u, &fail)) {
                fail = 1;
                break;
            }
            for (uint32_t c = 0; c < ga.n_chunks; c++) {
                Unit<kParts> x;
                if (kLeaf && scaled) times_leaf(f, factor, tkd + c * kKq + 8u * h);
                split_fetch<kParts>(f, x);
                if (loads && c + 1u < ga.n_chunks) fetch8<false>(f, src, koff + (c + 1u) * kKq);
                if (active) store_b_interleaved<NT, kParts>(sB + c * kBChunk, x, col, h);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            warp_arrive(smem_u32(&bfull_bar));
            t = (grp + 1u) << ga.mt_bits;   // the next column tile's first row tile
            cur.next_group(ga);
        }
    } else if (warp < kEpiWarp) {
        regs_dec<Regs<NT>::kBsIssue>();
        if (warp == kMmaWarp && lane == 0) {
            constexpr uint32_t idesc = mma_idesc<kParts>(NT);
            const uint32_t group = min(kParts == 2 && !kRuns ? 4u : group_chunks<kParts>(), ga.n_chunks), runs = ga.n_chunks >> ga.run_bits;
            RingPos ring;
            uint32_t j = 0, gi = 0;
            bool ok = true;
            for (uint64_t t = t0; t < t1 && !fail && ok; t++, j++) {
                const uint64_t grp = t >> ga.mt_bits;
                if (t == t0 || (t & (ga.n_mt - 1u)) == 0u) {   // a new column tile: its B is loaded
                    if (!wait_or_fail(smem_u32(&bfull_bar), gi & 1u, &fail)) {
                        ok = false;
                        break;
                    }
                    gi++;
                }
                for (uint32_t c = 0; c < ga.n_chunks && ok; c += group) {
                    const uint32_t run = c >> ga.run_bits, at = kRuns ? c & ((1u << ga.run_bits) - 1u) : c;
                    const RunSlot<NA> slot(j, run, runs);
                    const bool starts = at == 0u, ends = kRuns ? run != 0u && at + group == 1u << ga.run_bits : c + group >= ga.n_chunks;
                    const uint32_t buf = kRuns ? slot.buf : j % NA;
                    if (starts) {
                        ok = wait_or_fail(smem_u32(&acce_bar[buf]), ((kRuns ? slot.uses : j / NA) & 1u) ^ 1u, &fail);
                        if (!ok) break;
                        tc_fence_after();
                    }
                    auto b_at = [&](uint32_t i, uint32_t, uint32_t (&bs)[2][kParts]) {
                        const uint32_t sb = smem_u32(sB) + (c + i) * kBChunk;
#pragma unroll
                        for (uint32_t q = 0; q < (uint32_t)kParts; q++) {
                            bs[0][q] = sb + q * kRegB;
                            bs[1][q] = sb + (kParts + q) * kRegB;
                        }
                    };
                    ok = mma_group<kParts>(tmem + buf * kCols, group, starts, ring, S, sbase, kStage, kRegA, full_bar, empty_bar, b_at,
                                           idesc, &fail);
                    if (ok && ends) mma_commit(smem_u32(&accf_bar[buf]));
                }
                if (!ok) break;
                // the column tile's last row tile in this range: its B regions may be reloaded
                // once these MMAs have completed
                if (t + 1u == t1 || ((t + 1u) >> ga.mt_bits) != grp) mma_commit(smem_u32(&bempty_bar));
            }
            if (!ok) fail = 1;
            mma_commit(smem_u32(&drain_bar));
            if (!mbar_wait(smem_u32(&drain_bar), 0, kPolls)) fail = 1;
        }
        __syncwarp();
    } else {
        if constexpr (Regs<NT>::kBsEpi > Regs<NT>::kLaunch) regs_inc<Regs<NT>::kBsEpi>();
        else regs_dec<Regs<NT>::kBsEpi>();
        const uint32_t q = warp & 3u, lanes = tmem + ((q * 32u) << 16);
        const uint32_t runs = ga.n_chunks >> ga.run_bits;
        constexpr uint32_t kSum = kW < 16u ? kW : 16u;   // columns added at a time
        const uint32_t share = (warp - kEpiWarp) >> 2;
        uint32_t j = 0;
        BsCursor cur;
        cur.c = tile_coord_bs(t0, ga);
        bool ok = true;
        // this lane's row of C in a tile
        auto row_of = [&](const TileCoord &tc) {
            return ga.arenas + (uint64_t)tc.il * ga.a.arena_elems + g.c_off + pext_runs(tc.beta, g.cb, g.n_cb) +
                   pext_runs(tc.mt * kRows + 32u * q + lane, g.cm, g.n_cm);
        };
        uint32_t coff[kW / 2u];   // offsets of a block's columns in C
#pragma unroll
        for (uint32_t i = 0; i < kW / 2u; i++) coff[i] = pext_runs(i, g.cn, g.n_cn);
        for (uint64_t t = t0; t < t1; t++, j++, cur.next(ga)) {
            const TileCoord &tc = cur.c;
            const RunSlot<NA> last(j, runs - 1u, runs);
            const uint32_t buf = kRuns ? last.buf : j % NA;
            float2 *Crow = row_of(tc);   // while the MMAs run
            Unscale un{1.f, 1.f, false};
            if (kParts == 2) un = unscale_of(side_max<kLeaf>(ga, true, tc.il), side_max<kLeaf>(ga, false, tc.il));
            uint32_t largest = 0;
            if constexpr (kRuns) {
                for (uint32_t r = 1; r + 1u < runs && ok; r++) {
                    ok = warp_wait_or_fail(smem_u32(&accf_bar[buf]), RunSlot<NA>(j, r, runs).uses & 1u, &fail);
                    if (!ok) break;
                    tc_fence_after();
                    for (uint32_t j0 = share * kSum; j0 < (uint32_t)NT; j0 += 2u * kSum)
                        tmem_add<kSum>(lanes + (buf - 1u) * kCols + j0, lanes + buf * kCols + j0);
                    tc_fence_before();
                    warp_arrive(smem_u32(&acce_bar[buf]));
                }
            }
            if (ok) ok = warp_wait_or_fail(smem_u32(&accf_bar[buf]), (kRuns ? last.uses : j / NA) & 1u, &fail);
            if (!ok) break;
            tc_fence_after();
            const uint32_t taddr = lanes + buf * kCols;
            for (uint32_t j0 = share * kW; j0 < (uint32_t)NT; j0 += 2u * kW) {
                float2 *Cblk = Crow + pext_runs(tc.nt * kNc + j0 / 2u, g.cn, g.n_cn);
                uint32_t r[kW];
                tmem_ld_pairs<kW>(taddr + j0, r);
                if constexpr (kRuns) add_columns<kW>(r, taddr - kCols + j0);
#pragma unroll
                for (uint32_t i = 0; i < kW / 2u; i++) {
                    const float2 c = kParts == 2 ? unscaled(un, r[2u * i], r[2u * i + 1u])
                                                 : make_float2(__uint_as_float(r[2u * i]), __uint_as_float(r[2u * i + 1u]));
                    Cblk[coff[i]] = c;
                    if (ga.max_c) largest = abs_max(largest, c);
                }
            }
            tc_fence_before();
            warp_arrive(smem_u32(&acce_bar[buf]));
            if (kRuns) warp_arrive(smem_u32(&acce_bar[buf - 1u]));
            if (ga.max_c) note_max_warp(ga.max_c + tc.il, largest);
        }
        if (!ok) fail = 1;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(NA * kCols) : "memory");
    }
    if (fail && threadIdx.x == 0) atomicCAS(ga.a.status, 0u, 4u /* QVX_ETIMEOUT */);
}

}  // namespace

// Grid of a persistent tensor-core kernel: the SM count times the CTAs an SM holds (within
// its 512 tensor-memory columns, so that no allocation ever waits for another CTA's
// columns), queried once per device and kernel (under a lock: host threads may launch on
// several streams at once).
template <int NT, int kParts, bool kBs, bool kLeaf, bool kRuns>
static cudaError_t gemm_grid(uint64_t n_tiles, uint64_t *grid) {
    static int per_sm[64] = {0}, sms[64] = {0};
    static std::mutex mu;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!per_sm[dev]) {
        const void *fn = kBs ? reinterpret_cast<const void *>(gemm_tc_bs_kernel<NT, kParts, kLeaf, kRuns>)
                             : reinterpret_cast<const void *>(gemm_tc_kernel<NT, kParts, kLeaf, kRuns>);
        const size_t smem = kBs ? (size_t)kBsBytes : smem_bytes<NT, kParts>(n_stages<kParts>(4u), 1024);
        const int threads = (int)block_threads<NT>();
        if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
            return e;
        cudaFuncAttributes fa;
        if ((e = cudaFuncGetAttributes(&fa, fn)) != cudaSuccess) return e;
        // the roles' register shares must fit in what the block is launched with
        if ((uint32_t)fa.numRegs != Regs<NT>::kLaunch) return cudaErrorInvalidConfiguration;
        int n = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, smem)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        const int cols = (int)((kBs || kRuns ? bs_accs<NT>() : 2u) * acc_cols<NT>());
        per_sm[dev] = n < 1 ? -1 : std::min(n, 512 / cols);
    }
    if (per_sm[dev] < 1) return cudaErrorInvalidConfiguration;
    *grid = std::min<uint64_t>(n_tiles, (uint64_t)sms[dev] * (uint64_t)per_sm[dev]);
    return cudaSuccess;
}

template <int NT, int kParts, bool kLeaf, bool kRuns>
static cudaError_t launch_gemm_nt(GemmArgs ga, cudaStream_t s) {
    ga.n_tiles = ((uint64_t)ga.n_items << ga.g.nb) * ga.n_mt * ga.n_nt;
    if (ga.n_tiles == 0) return cudaErrorInvalidConfiguration;
    uint64_t grid = 0;
    cudaError_t e;
    // B-stationary form: B's regions of every chunk stay resident, and at least 4 row tiles per
    // column tile reuse them (with 2, the reload between column tiles, which waits for the old
    // tile's MMAs, cost more than the reuse saved; tile coordinates above the row tiles within
    // 32 bits)
    if (ga.n_chunks <= bs_chunks<NT, kParts>() && ga.n_mt >= 4u && (uint64_t)ga.n_items * ga.n_nt < (1ull << 32)) {
        if ((e = gemm_grid<NT, kParts, true, kLeaf, kRuns>(ga.n_tiles, &grid)) != cudaSuccess) return e;
        ga.stages = bs_stages<NT, kParts>(ga.n_chunks);
        // Shared memory asked for leaves the rest of the SM's 256 KB as L1 cache. At 256 columns
        // and up to 32 summed entries the step is bound by C's stores, and the smallest cache
        // serves it best (s120 of circuit 5002: 3.05 ms with 222 KB asked for, 3.42 with the
        // 174 KB used; s125 of 5001 6.33 and 7.20). The others read A's rows through the cache:
        // they ask for what they use (narrow steps 10 % faster than with 222 KB), with three
        // stages from 64 summed entries (s118 of 5001 1.88 ms, 2.02 with five stages).
        size_t bytes = kBsBytes;
        if (NT < 256 || ga.n_chunks > 2u) {
            if (NT >= 256) ga.stages = kParts == 2 ? 4u : 3u;
            bytes = ga.stages * a_bytes<kParts>() + ga.n_chunks * (bs_b_bytes<NT, kParts>() + 12u * kKq);
        }
        gemm_tc_bs_kernel<NT, kParts, kLeaf, kRuns><<<(unsigned)grid, block_threads<NT>(), bytes, s>>>(ga);
        return cudaGetLastError();
    }
    // dynamic shared memory: the operand stage ring and the summed index tables, sized for the largest
    // summed index (1024 entries)
    if ((e = gemm_grid<NT, kParts, false, kLeaf, kRuns>(ga.n_tiles, &grid)) != cudaSuccess) return e;
    gemm_tc_kernel<NT, kParts, kLeaf, kRuns><<<(unsigned)grid, (int)block_threads<NT>(), smem_bytes<NT, kParts>(n_stages<kParts>(ga.n_chunks), 1024), s>>>(ga);
    return cudaGetLastError();
}

template <int kParts, bool kLeaf>
static cudaError_t launch_gemm_split(const GemmArgs &ga, uint32_t nt_cols, cudaStream_t s) {
    if constexpr (kParts == 2) {
        // Up to four chunks are one group. Longer sums take runs of two chunks up to 128 summed entries, of
        // four beyond, where two cost 8 to 20 % more (512 entries: 2.18 and 2.01 ms; 2.04 in one
        // accumulator) for half the truncations.
        static_assert(bs_stages<256, 2>(4u) >= 4u && bs_stages<128, 2>(4u) >= 4u, "a group of four");
        GemmArgs gr = ga;
        gr.run_bits = ga.n_chunks > 8u ? 2u : 1u;
        if (ga.n_chunks >= 8u) switch (nt_cols) {
            case 16: return launch_gemm_nt<16, kParts, kLeaf, true>(gr, s);
            case 32: return launch_gemm_nt<32, kParts, kLeaf, true>(gr, s);
            case 64: return launch_gemm_nt<64, kParts, kLeaf, true>(gr, s);
            case 128: return launch_gemm_nt<128, kParts, kLeaf, true>(gr, s);
            default: return launch_gemm_nt<256, kParts, kLeaf, true>(gr, s);
        }
    }
    switch (nt_cols) {
        case 16: return launch_gemm_nt<16, kParts, kLeaf, false>(ga, s);
        case 32: return launch_gemm_nt<32, kParts, kLeaf, false>(ga, s);
        case 64: return launch_gemm_nt<64, kParts, kLeaf, false>(ga, s);
        case 128: return launch_gemm_nt<128, kParts, kLeaf, false>(ga, s);
        default: return launch_gemm_nt<256, kParts, kLeaf, false>(ga, s);
    }
}

}  // namespace qvx

// A tensor-core contraction fused with the reduction of its result (stepwise engine,
// opts.tensor_cores, fp16 parts): X[b, m, n] = sum_k A B, then E = sum_J X D, where D is another
// tensor over modes of X and J are modes of X (any of b, m, n) that only D shares. X is the
// largest tensor of such a program (34 GB of the 125 GB that circuit 5001's step list moves) and
// is read exactly once, so its tiles are multiplied by D and summed while they leave tensor
// memory, and X never reaches memory.
//
// Layout of the work: a tile's 128 rows (tensor-memory lanes) are row modes that stay in E, its
// 128 columns are column modes with up to four of J lowest, so a lane sums its J columns in
// registers. The rest of J (jo) is walked tile by tile into the same registers; E is stored when
// all of J is summed. A unit fixes everything else but the remaining row modes (mo), so one
// unit keeps its B (for every value of those jo bits that B holds) in shared memory, as the
// B-stationary form does. Units that differ only in modes that D lacks run next to each other
// on different SMs and read D's entries through L2 together.
//
// Roles are those of the B-stationary form (gemm_tc.cuh). The epilogue holds its accumulators,
// a block's columns and two blocks' D entries in registers, so it takes most of the register
// file. What bounds it is the latency of D's entries: 128 KB per tile with 32 to 64 KB in
// flight per SM (DRAM 19 %, tensor pipe 18 %, LSU data pipe 19 % busy). Circuit 5001: 7.02 ms,
// the two steps before 6.22 + 5.84; circuit 5002: 4.6 ms, before 3.64 + 3.12.
#include "gemm_tc.cuh"

namespace qvx {
namespace {

constexpr uint32_t kNt = 256u;                    // real columns of a tile (128 complex)
constexpr uint32_t kRBThreads = 128u;             // B producers: two units each
constexpr uint32_t kRMmaWarp = (256u + kRBThreads) / 32u;
constexpr uint32_t kREpiWarp = kRMmaWarp + 4u;
constexpr uint32_t kRThreads = 32u * kREpiWarp + kEpiThreads;
constexpr uint32_t kRLaunchRegs = 80u, kRRegsA = 72u, kRRegsB = 56u, kRRegsIssue = 24u, kRRegsEpi = 128u;
static_assert(256u * kRRegsA + kRBThreads * kRRegsB + 128u * kRRegsIssue + 256u * kRRegsEpi <= kRLaunchRegs * kRThreads,
              "register shares");
constexpr uint32_t kRStages = 3u;
constexpr uint32_t kRegionA = region_bytes(kRows), kRegionB = region_bytes(kNt);
constexpr uint32_t kRStage = a_bytes<2>(), kRChunkB = 4u * kRegionB;

struct ReduceArgs {
    LaunchArgs a;
    ReduceStep r;
    GemmScale sc;
    uint32_t *max_c;
    int64_t item0, n_items;
    float2 *arenas;
    uint32_t n_chunks;
    uint64_t n_units;
};

__device__ __forceinline__ uint32_t mv(uint32_t idx, const ModeMap &m) { return pext_runs(idx, m.runs, m.n); }

template <int JC>   // columns of a tile that are summed: 2^JC neighbouring ones
__global__ void __launch_bounds__(kRThreads, 1) gemm_tc_reduce_kernel(ReduceArgs ra) {
    constexpr uint32_t S = kRStages;
    extern __shared__ __align__(1024) unsigned char gsm[];
    __shared__ __align__(8) uint64_t full_bar[S], empty_bar[S], accf_bar[2], acce_bar[2], bfull_bar, bempty_bar, drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int fail;
    const ReduceStep &r = ra.r;
    const uint32_t warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t sbase = smem_u32(gsm);
    unsigned char *sB = gsm + S * kRStage;
    const uint32_t K = ra.n_chunks * kKq, n_jb = 1u << r.jb, n_jm = 1u << (r.jo - r.jb), n_mo = 1u << r.mo;
    uint32_t *tka = reinterpret_cast<uint32_t *>(sB + n_jb * ra.n_chunks * kRChunkB);
    uint32_t *tkb = tka + K;
    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < S; s++) {
            mbar_init(smem_u32(&full_bar[s]), 8);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        for (uint32_t b = 0; b < 2; b++) {
            mbar_init(smem_u32(&accf_bar[b]), 1);
            mbar_init(smem_u32(&acce_bar[b]), kEpiThreads / 32u);
        }
        mbar_init(smem_u32(&bfull_bar), kRBThreads / 32u);
        mbar_init(smem_u32(&bempty_bar), 1);
        mbar_init(smem_u32(&drain_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fail = 0;
    }
    if (warp == kRMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(2u * kNt)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (uint32_t i = threadIdx.x; i < K; i += kRThreads) {
        tka[i] = mv(i, r.k_a);
        tkb[i] = mv(i, r.k_b);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const bool k8 = (1u << r.nk) < kKq;   // 8 summed entries: the second half of the chunk is zero
    const uint32_t unit_mask = (uint32_t)((1ull << r.nu) - 1ull);
    if (warp < 8u) {
        regs_dec<kRRegsA>();
        // A producers: row u & 127 of the tile, summed half u >> 7; tiles unit by unit, mo, jo
        const uint32_t row = threadIdx.x & 127u, h = threadIdx.x >> 7;
        const bool loads = !(k8 && h == 1u);
        const uint32_t *koff = tka + 8u * h;
        const uint32_t own = mv(row, r.row_a);
        uint64_t u = blockIdx.x;
        uint32_t mo = 0, jo = 0, c = 0, item_max = 0;
        const float2 *base = nullptr, *src = nullptr;
        auto setup_unit = [&]() {
            const int64_t il = (int64_t)(u >> r.nu);
            const float2 *arena = ra.arenas + (uint64_t)il * ra.a.arena_elems;
            base = gemm_operand(ra.a, arena, r.a_off, r.flags & kStepALeaf, ra.item0 + il) + mv((uint32_t)u & unit_mask, r.unit_a) + own;
            item_max = operand_max(ra.sc.max_a, ra.sc.leaf_max_a, il);
        };
        auto setup_tile = [&]() { src = base + mv(mo, r.mo_a) + mv(jo, r.jo_a); };
        auto fetch = [&](Fetch &f) {
            if (u >= ra.n_units) return;
            if (loads) fetch8<false>(f, src, koff + c * kKq);
            f.max = item_max;
            if (++c < ra.n_chunks) return;
            c = 0;
            if (++jo == n_jb * n_jm) {
                jo = 0;
                if (++mo == n_mo) {
                    mo = 0;
                    u += gridDim.x;
                    if (u >= ra.n_units) return;
                    setup_unit();
                }
            }
            setup_tile();
        };
        setup_unit();
        setup_tile();
        const uint64_t units = (ra.n_units - blockIdx.x + gridDim.x - 1) / gridDim.x;
        const uint64_t total = (units * ra.n_chunks) << (r.mo + r.jo);
        RingPos ring;
        auto produce = [&](Fetch &f) -> bool {
            Unit<2> x;
            split_fetch<2>(f, x);
            fetch(f);
            if (!warp_wait_or_fail(smem_u32(&empty_bar[ring.s]), ring.phase ^ 1u, &fail)) {
                fail = 1;
                return false;
            }
            store_a<2>(gsm + ring.s * kRStage, x, row, h);
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
    } else if (warp < kRMmaWarp) {
        regs_dec<kRRegsB>();
        // B producers: complex column v of both summed halves; per unit, every chunk for every
        // value of the jo bits that B holds
        const uint32_t col = threadIdx.x - 256u;
        const uint32_t own = mv(col, r.col_b);
        uint32_t gi = 0;
        for (uint64_t u = blockIdx.x; u < ra.n_units; u += gridDim.x, gi++) {
            const int64_t il = (int64_t)(u >> r.nu);
            const float2 *arena = ra.arenas + (uint64_t)il * ra.a.arena_elems;
            const float2 *base = gemm_operand(ra.a, arena, r.b_off, r.flags & kStepBLeaf, ra.item0 + il) +
                                 mv((uint32_t)u & unit_mask, r.unit_b) + own;
            Fetch f;
            fetch_zero(f);
            f.max = operand_max(ra.sc.max_b, ra.sc.leaf_max_b, il);
            fetch8<false>(f, base, tkb);   // the first entries, while the old unit's last MMAs run
            if (!warp_wait_or_fail(smem_u32(&bempty_bar), (gi & 1u) ^ 1u, &fail)) {
                fail = 1;
                break;
            }
            for (uint32_t jb = 0; jb < n_jb; jb++) {
                for (uint32_t ch = 0; ch < 2u * ra.n_chunks; ch++) {   // chunk and half
                    Unit<2> x;
                    split_fetch<2>(f, x);
                    uint32_t nb = jb, nch = ch + 1u;
                    if (nch == 2u * ra.n_chunks) {
                        nch = 0;
                        nb++;
                    }
                    if (nb < n_jb) {
                        if (k8 && nch == 1u) {
                            const uint32_t m = f.max;
                            fetch_zero(f);
                            f.max = m;
                        } else {
                            fetch8<false>(f, base + mv(nb * n_jm, r.jo_b), tkb + 8u * nch);
                        }
                    }
                    store_b_interleaved<kNt, 2>(sB + (jb * ra.n_chunks + (ch >> 1)) * kRChunkB, x, col, ch & 1u);
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            warp_arrive(smem_u32(&bfull_bar));
        }
    } else if (warp < kREpiWarp) {
        regs_dec<kRRegsIssue>();
        if (warp == kRMmaWarp && lane == 0) {
            constexpr uint32_t idesc = mma_idesc<2>(kNt);
            const uint32_t group = min(group_chunks<2>(), ra.n_chunks);
            RingPos ring;
            uint32_t j = 0, gi = 0;
            bool ok = true;
            for (uint64_t u = blockIdx.x; u < ra.n_units && ok; u += gridDim.x, gi++) {
                if (!wait_or_fail(smem_u32(&bfull_bar), gi & 1u, &fail)) {
                    ok = false;
                    break;
                }
                const uint32_t tiles = n_mo << r.jo;
                for (uint32_t t = 0; t < tiles && ok; t++, j++) {
                    const uint32_t buf = j & 1u;
                    if (!wait_or_fail(smem_u32(&acce_bar[buf]), ((j >> 1) & 1u) ^ 1u, &fail)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t d = tmem + buf * kNt;
                    // jo = jb * n_jm + jm: the B of this tile's jb
                    const uint32_t b0 = ((t & (n_jb * n_jm - 1u)) >> (r.jo - r.jb)) * ra.n_chunks;
                    for (uint32_t c = 0; c < ra.n_chunks && ok; c += group) {
                        auto b_at = [&](uint32_t i, uint32_t, uint32_t (&bs)[2][2]) {
                            const uint32_t sb = smem_u32(sB) + (b0 + c + i) * kRChunkB;
                            bs[0][0] = sb;
                            bs[0][1] = sb + kRegionB;
                            bs[1][0] = sb + 2u * kRegionB;
                            bs[1][1] = sb + 3u * kRegionB;
                        };
                        ok = mma_group<2>(d, group, c == 0u, ring, S, sbase, kRStage, kRegionA, full_bar, empty_bar, b_at, idesc, &fail);
                    }
                    if (ok) mma_commit(smem_u32(&accf_bar[buf]));
                }
                if (ok) mma_commit(smem_u32(&bempty_bar));   // the unit's B may be replaced after these MMAs
            }
            if (!ok) fail = 1;
            mma_commit(smem_u32(&drain_bar));
            if (!mbar_wait(smem_u32(&drain_bar), 0, kPolls)) fail = 1;
        }
        __syncwarp();
    } else {
        regs_inc<kRRegsEpi>();
        // epilogue: warp w holds rows 32 (w mod 4) + lane; the two warps of a lane quarter take
        // alternate blocks of 16 columns, 16 >> JC entries of E each
        constexpr uint32_t kE = 16u >> JC;
        const uint32_t q = warp & 3u, share = (warp - kREpiWarp) >> 2;
        const uint32_t own_d = mv(32u * q + lane, r.row_d), own_e = mv(32u * q + lane, r.row_e);
        uint32_t doff[16];
#pragma unroll
        for (uint32_t i = 0; i < 16u; i++) doff[i] = mv(i, r.col_d);
        // tile cursor of D: a block's entries are loaded while the block before is summed (without
        // that the merged step of circuit 5001 took 7.33 instead of 7.02 ms; with prefetches of
        // D into L2 a tile ahead 8.6 ms by line, 16.6 ms by bulk prefetch of row runs)
        uint64_t pu = blockIdx.x;
        uint32_t pmo = 0, pjo = 0;
        const float2 *pbase = nullptr;
        auto d_unit = [&]() {
            const int64_t il = (int64_t)(pu >> r.nu);
            pbase = gemm_operand(ra.a, ra.arenas + (uint64_t)il * ra.a.arena_elems, r.d_off, r.flags & kReduceDLeaf, ra.item0 + il) +
                    mv((uint32_t)pu & unit_mask, r.unit_d);
        };
        auto d_tile = [&]() { return pbase + mv(pmo, r.mo_d) + mv(pjo, r.jo_d); };
        auto d_next = [&]() {   // past the last tile the cursor stays on it
            if (++pjo < n_jb * n_jm) return;
            pjo = 0;
            if (++pmo < n_mo) return;
            pmo = 0;
            if (pu + gridDim.x < ra.n_units) {
                pu += gridDim.x;
                d_unit();
            }
        };
        auto load_block = [&](float2 (&dv)[16], const float2 *dt, uint32_t b) {
            const float2 *db = dt + mv((share + 2u * b) * 16u, r.col_d) + own_d;
#pragma unroll
            for (uint32_t i = 0; i < 16u; i++) dv[i] = db[doff[i]];
        };
        d_unit();
        const float2 *dt = d_tile();   // the tile that is summed
        float2 dv[2][16];
        load_block(dv[0], dt, 0);
        uint32_t j = 0;
        bool ok = true;
        for (uint64_t u = blockIdx.x; u < ra.n_units && ok; u += gridDim.x) {
            const int64_t il = (int64_t)(u >> r.nu);
            float2 *ebase = ra.arenas + (uint64_t)il * ra.a.arena_elems + r.e_off + mv((uint32_t)u & unit_mask, r.unit_e) + own_e;
            uint32_t largest = 0;
            for (uint32_t mo = 0; mo < n_mo && ok; mo++) {
                float2 acc[4][kE];
#pragma unroll
                for (uint32_t b = 0; b < 4u; b++)
#pragma unroll
                    for (uint32_t e = 0; e < kE; e++) acc[b][e] = make_float2(0.f, 0.f);
                for (uint32_t jo = 0; jo < n_jb * n_jm; jo++, j++) {
                    const uint32_t buf = j & 1u;
                    const uint32_t taddr = tmem + ((q * 32u) << 16) + buf * kNt;
                    d_next();
                    const float2 *dn = d_tile();
                    if (!warp_wait_or_fail(smem_u32(&accf_bar[buf]), (j >> 1) & 1u, &fail)) {
                        fail = 1;
                        ok = false;
                        break;
                    }
                    tc_fence_after();
#pragma unroll
                    for (uint32_t b = 0; b < 4u; b++) {
                        load_block(dv[(b + 1u) & 1u], b < 3u ? dt : dn, (b + 1u) & 3u);
#pragma unroll
                        for (uint32_t half = 0; half < 2u; half++) {
                            uint32_t x[16];
                            tmem_ld_pairs<16>(taddr + 2u * ((share + 2u * b) * 16u + 8u * half), x);
#pragma unroll
                            for (uint32_t i = 0; i < 8u; i++) {
                                const float xr = __uint_as_float(x[2u * i]), xi = __uint_as_float(x[2u * i + 1u]);
                                const float2 d = dv[b & 1u][8u * half + i];
                                float2 &s = acc[b][(8u * half + i) >> JC];
                                s.x = fmaf(xr, d.x, s.x);
                                s.x = fmaf(-xi, d.y, s.x);
                                s.y = fmaf(xr, d.y, s.y);
                                s.y = fmaf(xi, d.x, s.y);
                            }
                        }
                    }
                    tc_fence_before();
                    warp_arrive(smem_u32(&acce_bar[buf]));
                    dt = dn;
                }
                if (!ok) break;
                const Unscale un = unscale_of(operand_max(ra.sc.max_a, ra.sc.leaf_max_a, il),
                                              operand_max(ra.sc.max_b, ra.sc.leaf_max_b, il));
                float2 *emo = ebase + mv(mo, r.mo_e);
#pragma unroll
                for (uint32_t b = 0; b < 4u; b++)
#pragma unroll
                    for (uint32_t e = 0; e < kE; e++) {
                        const uint32_t kept = ((share + 2u * b) * 16u >> JC) + e;   // kept column index
                        float2 v = make_float2(acc[b][e].x * un.f1, acc[b][e].y * un.f1);
                        if (un.two) v = make_float2(v.x * un.f2, v.y * un.f2);
                        emo[mv(kept, r.col_e)] = v;
                        if (ra.max_c) largest = abs_max(largest, v);
                    }
            }
            if (ok && ra.max_c) note_max_warp(ra.max_c + il, largest);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kRMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2u * kNt) : "memory");
    }
    if (fail && threadIdx.x == 0) atomicCAS(ra.a.status, 0u, 4u /* QVX_ETIMEOUT */);
}

template <int JC>
cudaError_t launch_jc(const ReduceArgs &ra, size_t bytes, cudaStream_t s) {
    static int sms[64] = {0};
    static std::mutex mu;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int n_sm = 0;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!sms[dev]) {
            cudaFuncAttributes fa;
            if ((e = cudaFuncGetAttributes(&fa, gemm_tc_reduce_kernel<JC>)) != cudaSuccess) return e;
            if ((uint32_t)fa.numRegs != kRLaunchRegs) return cudaErrorInvalidConfiguration;   // the roles' shares
            if ((e = cudaFuncSetAttribute(gemm_tc_reduce_kernel<JC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBsBytes)) !=
                cudaSuccess)
                return e;
            if ((e = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        }
        n_sm = sms[dev];
    }
    const unsigned grid = (unsigned)std::min<uint64_t>(ra.n_units, (uint64_t)n_sm);
    gemm_tc_reduce_kernel<JC><<<grid, kRThreads, bytes, s>>>(ra);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_reduce_step(const LaunchArgs &a, const ReduceStep &r, const GemmScale &scale, uint32_t *max_c,
                               int64_t item0, int64_t n_items, float2 *arenas, cudaStream_t s) {
    ReduceArgs ra;
    ra.a = a;
    ra.r = r;
    ra.sc = scale;
    ra.max_c = max_c;
    ra.item0 = item0;
    ra.n_items = n_items;
    ra.arenas = arenas;
    ra.n_chunks = std::max(1u, (1u << r.nk) / kKq);
    ra.n_units = (uint64_t)n_items << r.nu;
    const size_t bytes = kRStages * kRStage + ((size_t)ra.n_chunks << r.jb) * kRChunkB + 8u * kKq * ra.n_chunks;
    if (n_items <= 0 || r.nk < 3 || r.nu > 31 || bytes > kBsBytes) return cudaErrorInvalidConfiguration;
    switch (r.jc) {
        case 2: return launch_counted(launch_jc<2>(ra, bytes, s));
        case 3: return launch_counted(launch_jc<3>(ra, bytes, s));
        case 4: return launch_counted(launch_jc<4>(ra, bytes, s));
        default: return cudaErrorInvalidConfiguration;
    }
}

}  // namespace qvx

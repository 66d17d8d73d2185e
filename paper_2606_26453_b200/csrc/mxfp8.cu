// Block-scaled FP8 (MXFP8) twins of the six grouped GEMMs (gate/up forward, down forward, down dgrad, gate/up dgrad, and
// the two weight gradients, further down) on the block-scaled tensor-core path (tcgen05.mma kind::mxf8f6f4 with block_scale): quantisers, one GEMM
// in two tilings, and the SwiGLU activation with the activation quantiser fused in.  Every GEMM here is
//   out[r, :] = dequant(a row r) . dequant(b[e])^T   for the rows r of expert e,
// a [R, k] and b [E, n_feat, k] both contraction-contiguous; the callers choose which tensors play a and b.
//
// Format: E4M3 elements, one E8M0 scale (a power of two, 2^(s-127)) per 32 consecutive elements along the
// contraction; scale of a block with largest magnitude a > 0: 2^(floor(log2 a) - 8); elements = v / scale rounded to
// nearest even, saturating at 448; an all-zero block: s = 0 and zero codes.  The decisions that produce integers
// (scale byte, element code) are taken on exact values on both sides of the parity test: the inputs are bf16, the
// division by a power of two is exact in fp32, and the FP8 conversion instruction rounds to nearest even.
//
// Layouts (chosen so that the GEMM's scale factors reach tensor memory without per-element work):
//   activation codes   [R, k] bytes, contraction contiguous
//   activation scales  [k/128][R] 32-bit words: the 4 scale bytes of the 4 blocks of 32 inside one 128-wide slice of
//                      the contraction, for one row -- rows of a tile start anywhere, so a warp gathers 128 words per
//                      K slice and lays them out for the tensor-memory copy
//   weight codes       [E, n_feat, k] bytes, contraction contiguous (weights stored feature-contiguous are transposed by
//                      their quantiser)
//   weight scales      first [E][n_feat/128][k/128][512 bytes]: per 128 output features x 128 contraction elements, byte
//                      (f % 32) * 16 + ((f % 128) / 32) * 4 + block -- the 32 x 16-byte pattern that
//                      tcgen05.cp.32x128b.warpx4 copies from shared memory into 4 tensor-memory columns (lane = f % 32,
//                      column = (f % 128) / 32, byte = block); then the same bytes in the tiling of the CTA-pair kernel
//                      (see there)
//
// Single-CTA kernel: one or two CTAs per SM, persistent over the same row-ragged tile list as the bf16 kernels (tiles of 128 or
// 64 rows x 128 output features), K slices of 128 (= 128 bytes per row: the same swizzled stage geometry as 64 bf16).
//   warp 0      TMA producer: A and B code tiles, bulk copy of the weight-scale block
//   warp 1      four tcgen05.mma (K = 32 each, scale byte k selected through the instruction descriptor), commit
//   warp 2      activation scales: gathers the tile's 128 words of the K slice and writes them in the copy's pattern
//   warps 3..6  epilogue: tcgen05.ld, round to bf16, staged bulk tensor stores
//   warp 7      tcgen05.cp of both scale blocks of a stage into tensor memory (with them the MMA thread took ~750
//               cycles per K slice, without ~580 of which it waits 110; that is fast enough for the weights to come at HBM rate)
// Accumulator double buffered; the scale blocks of a ring stage have 8 tensor-memory columns of their own.  Two forms of
// the kernel, see MxGeo.
#include <cuda_fp8.h>

#include "tc_ptx.cuh"

namespace moe {

__device__ int g_mx_status = 0;

#ifdef MOE_TEST_HOOKS
// Test-only build: when set, every producer leaves out the loads and the barrier arrival of its first ring stage, so that
// the bounded waits on that stage run out (see grouped_gemm.cu).
__device__ int g_mx_test_withhold_first_stage = 0;
extern "C" int moe_test_withhold_first_stage_mxfp8(int on) {
    return cudaMemcpyToSymbol(g_mx_test_withhold_first_stage, &on, sizeof(int)) == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}
#endif

int mx_read_and_clear_status(int* status_out) {
    int v = 0, zero = 0;
    if (cudaMemcpyFromSymbol(&v, g_mx_status, sizeof(int)) != cudaSuccess) return MOE_ERR_CUDA;
    if (v != 0 && cudaMemcpyToSymbol(g_mx_status, &zero, sizeof(int)) != cudaSuccess) return MOE_ERR_CUDA;
    *status_out = v;
    return MOE_OK;
}

namespace {

constexpr int MX_BM = 128, MX_BN = 128, MX_BK = 128;   // rows of a pair CTA's tile, features of a single-CTA tile, contraction elements per stage
constexpr int MX_MAX_STAGES = 6;
constexpr int MX_W_BYTES = MX_BN * MX_BK, MX_SF_BYTES = 512;
constexpr int MX_EPI_WARPS = 4;
constexpr int MX_COPY_WARP = 3 + MX_EPI_WARPS;   // the scale-copy warp comes after the epilogue warps
constexpr int MX_THREADS = 32 * (4 + MX_EPI_WARPS);
constexpr int MX_STAGING_BYTES = MX_EPI_WARPS * 2048;
constexpr int MX_MAX_E = 1024;
constexpr int MX_TMEM_COLS = 512;
constexpr int MX_SCALE_AHEAD = 4;   // K slices whose activation-scale words the scale warp keeps in flight
struct MxCtl {
    unsigned long long full[MX_MAX_STAGES];
    unsigned long long sf_full[MX_MAX_STAGES];   // the stage's scales are in tensor memory (and its operands landed)
    unsigned long long empty[MX_MAX_STAGES];
    unsigned long long tmem_full[2];
    unsigned long long tmem_empty[2];
    unsigned long long drain;
    unsigned long long drain_copy;
    uint32_t tmem_base;
    int abort_flag;
    // followed by int32_t offs[E + 1], tile_prefix[E + 1]
};
// The two forms of the single-CTA kernel, by the most rows of a tile (which of them runs: launch_mx_gemm).
//   128  rows on the M side of the MMA, 128 output features on the N side; one CTA per SM.
//   64   operand roles swapped: 128 output features on the M side, 64 rows on the N side, so that no stage carries rows of
//        other experts and both accumulators take 128 tensor-memory columns together; two CTAs per SM.
template <int ROWS>
struct MxGeo {
    static constexpr bool SWAPPED = ROWS < MX_BM;
    static constexpr int CTAS = SWAPPED ? 2 : 1;                // per SM
    static constexpr int STAGES = SWAPPED ? 4 : 6;
    static constexpr int TMEM_COLS = 512 / CTAS;
    static constexpr int SF_COL0 = 2 * ROWS;                    // scale slots after the two accumulators, 8 columns per stage
    static constexpr int X_BYTES = ROWS * MX_BK;
    static constexpr int SFX_OFF = MX_W_BYTES + X_BYTES, SFW_OFF = SFX_OFF + MX_SF_BYTES;
    static constexpr int STAGE_BYTES = SFW_OFF + MX_SF_BYTES;   // 25 KB, 33 KB
    static int smem_bytes(int E) {
        return STAGES * STAGE_BYTES + MX_STAGING_BYTES + 1024 + (int)sizeof(MxCtl) + 2 * (E + 1) * (int)sizeof(int32_t);
    }
    // an SM has 228 KB of shared memory, of which every CTA costs 1 KB more than it asks for
    static bool all_ctas_fit(int E) { return CTAS * (smem_bytes(E) + 1024) <= 228 * 1024; }
    static_assert(STAGES <= MX_MAX_STAGES && STAGE_BYTES % 1024 == 0 && SF_COL0 + STAGES * 8 <= TMEM_COLS, "stage layout");
};

struct MxParams {
    const int32_t* offsets;
    int E, k_tiles, n_tiles, n_cols;
    long long R;
    uint32_t x_bytes;     // that one load of activation codes delivers
    const uint32_t* sa;   // activation scale words [k_tiles][R]
    const uint8_t* sb;    // weight scale blocks [E][n_tiles][k_tiles][512]
    bf16* out;
    long long ldo;
};

// (roles in which a whole warp waits take the verdict through __all_sync: a wait that runs out for one lane while the
// barrier completes for another must not split the warp ahead of a warp-wide instruction)
__device__ __forceinline__ bool mx_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    return mbar_wait_status(bar, parity, abort_flag, &g_mx_status);
}

// K-major operand tile [rows][128 bytes], 128-byte swizzle: 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t mx_operand_desc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// Scale block [32 rows][16 bytes], no swizzle: 8-row groups 128 bytes apart.
__device__ __forceinline__ uint64_t mx_scale_desc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | (1ull << 16) | ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
}
// Instruction descriptor of the block-scaled kind: E4M3 x E4M3, both K-major, E8M0 scales, scale byte `sf` of the
// scale columns for both operands.
template <int ROWS>
__device__ __forceinline__ uint32_t mx_idesc(uint32_t sf) {   // M = 128, N = ROWS (128 features are as many as 128 rows)
    return (sf << 4) | ((uint32_t)(ROWS >> 3) << 17) | (1u << 23) | ((uint32_t)(MX_BN >> 4) << 24) | (sf << 29);
}
__device__ __forceinline__ void mx_copy_scales(uint32_t taddr, uint64_t sdesc) {
    asm volatile("tcgen05.cp.cta_group::1.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}
__device__ __forceinline__ void mx_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t sfa,
                                       uint32_t sfb, uint32_t accumulate) {
    asm volatile(
        "{ .reg .pred p; setp.ne.u32 p, %4, 0;"
        " tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale [%0], %1, %2, %3, [%5], [%6], p; }" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb)
        : "memory");
}

struct MxTile {
    int e, row0, row_end, n0;
};
template <int ROWS>
__device__ __forceinline__ MxTile mx_decode(const MxParams& p, const int32_t* offs, const int32_t* tile_prefix, long long t) {
    int lo = 0, hi = p.E;   // largest e with tile_prefix[e] * n_tiles <= t
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if ((long long)tile_prefix[mid] * p.n_tiles <= t) lo = mid; else hi = mid;
    }
    const int local = (int)(t - (long long)tile_prefix[lo] * p.n_tiles);
    const int m_tiles_e = tile_prefix[lo + 1] - tile_prefix[lo];
    MxTile tl;
    tl.e = lo;
    // column tile major inside an expert: the CTAs that run at the same time share the expert's weight tiles in L2
    const int nt = local / m_tiles_e, mt = local - nt * m_tiles_e;
    tl.row0 = offs[lo] + mt * ROWS;
    tl.row_end = min(offs[lo + 1], tl.row0 + ROWS);
    tl.n0 = nt * MX_BN;
    return tl;
}

template <int ROWS>
__global__ void __launch_bounds__(MX_THREADS, MxGeo<ROWS>::CTAS)
mx_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
               const __grid_constant__ CUtensorMap map_o, const MxParams p) {
    using G = MxGeo<ROWS>;
    constexpr int MX_STAGES = G::STAGES, MX_STAGE_BYTES = G::STAGE_BYTES;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* tiles_ptr = smem_raw + (tiles_base - smem_u32(smem_raw));
    MxCtl* ctl = reinterpret_cast<MxCtl*>(tiles_ptr + MX_STAGES * MX_STAGE_BYTES + MX_STAGING_BYTES);
    int32_t* offs = reinterpret_cast<int32_t*>(ctl + 1);   // sized by E: up to 486 experts two CTAs fit an SM
    int32_t* tile_prefix = offs + p.E + 1;
    volatile int* abort_flag = &ctl->abort_flag;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (uniform, and known to be)

    if (threadIdx.x == 0) {
        for (int s = 0; s < MX_STAGES; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 2);    // the producer's arrive (with the byte count) + the scale warp's
            mbar_init(smem_u32(&ctl->sf_full[s]), 1);
            mbar_init(smem_u32(&ctl->empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(&ctl->tmem_full[a]), 1);
            mbar_init(smem_u32(&ctl->tmem_empty[a]), MX_EPI_WARPS);
        }
        mbar_init(smem_u32(&ctl->drain), 1);
        mbar_init(smem_u32(&ctl->drain_copy), 1);
        ctl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_tmap(&map_a);
        prefetch_tmap(&map_b);
        prefetch_tmap(&map_o);
    }
    // everything above may run while the kernel before is still finishing; the schedule is derived from its output
    grid_dependency_wait();
    for (int e = threadIdx.x; e <= p.E; e += MX_THREADS) offs[e] = p.offsets[e];
    __syncthreads();
    if (warp == 0) exclusive_tile_prefix(offs, tile_prefix, p.E, ROWS, lane);
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                     "r"((uint32_t)G::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, ctl->tmem_base, 0);
    const long long n_tiles_total = (long long)__shfl_sync(0xffffffffu, tile_prefix[p.E], 0) * p.n_tiles;
    auto stage_base = [&](uint32_t s) { return tiles_base + s * MX_STAGE_BYTES; };

    if (warp == 0) {
        // ================= producer =================
        {   // the whole warp on uniform values, one elected lane issues (see the bf16 kernels)
            uint32_t stage = 0, phase = 0, issued = 0;
            bool ok = true;
            for (long long t = blockIdx.x; ok && t < n_tiles_total; t += gridDim.x) {
                MxTile tl = mx_decode<ROWS>(p, offs, tile_prefix, t);
                tl.e = __shfl_sync(0xffffffffu, tl.e, 0); tl.row0 = __shfl_sync(0xffffffffu, tl.row0, 0); tl.n0 = __shfl_sync(0xffffffffu, tl.n0, 0);
                const uint8_t* sb_tile = p.sb + ((long long)tl.e * p.n_tiles + tl.n0 / MX_BN) * p.k_tiles * MX_SF_BYTES;
                for (int kt = 0; kt < p.k_tiles; ++kt) {
                    if (!__all_sync(0xffffffffu, mx_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u, abort_flag))) { ok = false; break; }
#ifdef MOE_TEST_HOOKS
                    if (g_mx_test_withhold_first_stage != 0 && issued == 0) {
                        ++issued;
                        if (++stage == MX_STAGES) { stage = 0; phase ^= 1u; }
                        continue;
                    }
#endif
                    const uint32_t full = smem_u32(&ctl->full[stage]);
                    const uint32_t a_dst = stage_base(stage);
                    if (elect_one()) {
                        mbar_arrive_expect_tx(full, MX_W_BYTES + p.x_bytes + MX_SF_BYTES);
                        tma_load_2d(a_dst, &map_b, kt * MX_BK, tl.e * p.n_cols + tl.n0, full);
                        tma_load_2d(a_dst + MX_W_BYTES, &map_a, kt * MX_BK, tl.row0, full);
                        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                                         a_dst + G::SFW_OFF),
                                     "l"(sb_tile + (long long)kt * MX_SF_BYTES), "r"(MX_SF_BYTES), "r"(full)
                                     : "memory");
                    }
                    __syncwarp();
                    ++issued;
                    if (++stage == MX_STAGES) { stage = 0; phase ^= 1u; }
                }
            }
            if (!ok) {   // leave no bulk copy in flight: bounded wait for the copies issued into each stage
                const uint32_t n_wait = issued < (uint32_t)MX_STAGES ? issued : (uint32_t)MX_STAGES;
                uint32_t s = stage, ph = phase;
                for (uint32_t i = 0; i < n_wait; ++i) {
                    if (s == 0) { s = MX_STAGES - 1; ph ^= 1u; } else { --s; }
                    const unsigned long long t0 = global_timer_ns();
                    while (!mbar_try_wait(smem_u32(&ctl->full[s]), ph) && global_timer_ns() - t0 < WAIT_LIMIT_NS / 4) {}
                }
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer =================
        {
            uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0;
            bool ok = true;
            for (long long t = blockIdx.x; ok && t < n_tiles_total; t += gridDim.x) {
                if (!__all_sync(0xffffffffu, mx_wait(smem_u32(&ctl->tmem_empty[acc]), acc_phase ^ 1u, abort_flag))) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * ROWS;
                for (int kt = 0; kt < p.k_tiles; ++kt) {
                    if (!__all_sync(0xffffffffu, mx_wait(smem_u32(&ctl->sf_full[stage]), phase, abort_flag))) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t a_base = stage_base(stage);
                    const uint32_t sfw_t = tmem_base + G::SF_COL0 + stage * 8, sfx_t = sfw_t + 4;
                    const uint64_t w_desc = mx_operand_desc(a_base), x_desc = mx_operand_desc(a_base + MX_W_BYTES);
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < MX_BK / 32; ++k)
                            mx_mma(d_tmem, (G::SWAPPED ? w_desc : x_desc) + (uint64_t)((k * 32) >> 4),
                                   (G::SWAPPED ? x_desc : w_desc) + (uint64_t)((k * 32) >> 4), mx_idesc<ROWS>(k), G::SWAPPED ? sfw_t : sfx_t,
                                   G::SWAPPED ? sfx_t : sfw_t, (kt != 0 || k != 0) ? 1u : 0u);
                        tc_commit<false>(smem_u32(&ctl->empty[stage]));
                    }
                    __syncwarp();
                    if (++stage == MX_STAGES) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                if (elect_one()) tc_commit<false>(smem_u32(&ctl->tmem_full[acc]));
                __syncwarp();
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
            // all issued MMAs must have retired before tensor memory is released
            if (elect_one()) {
                tc_commit_local<false>(smem_u32(&ctl->drain));
                const unsigned long long t0 = global_timer_ns();
                while (!mbar_try_wait(smem_u32(&ctl->drain), 0) && global_timer_ns() - t0 < WAIT_LIMIT_NS) {}
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // ================= activation scales =================
        // lane l owns rows l, 32 + l, 64 + l, 96 + l of the tile: one 16-byte piece of the 32 x 16-byte block
        uint32_t stage = 0, phase = 0;
        bool ok = true;
        for (long long t = blockIdx.x; ok && t < n_tiles_total; t += gridDim.x) {
            const MxTile tl = mx_decode<ROWS>(p, offs, tile_prefix, t);
            long long rows[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const long long r = (long long)tl.row0 + 32 * i + lane;
                rows[i] = r < p.R ? r : p.R - 1;   // rows past the end are never stored; any valid address will do
            }
            // the words of MX_SCALE_AHEAD slices are in flight at any time: one slice per global-load round trip would
            // bound the whole pipeline (the loads wait behind the operand traffic)
            auto load_slice = [&](int kt) {
                const uint32_t* s = p.sa + (long long)kt * p.R;
                uint4 w = make_uint4(__ldg(s + rows[0]), 0u, 0u, 0u);
                if (ROWS > 32) w.y = __ldg(s + rows[1]);
                if (ROWS > 64) { w.z = __ldg(s + rows[2]); w.w = __ldg(s + rows[3]); }
                return w;
            };
            uint4 q[MX_SCALE_AHEAD];
#pragma unroll
            for (int i = 0; i < MX_SCALE_AHEAD; ++i) q[i] = load_slice(min(i, p.k_tiles - 1));
            for (int kt0 = 0; ok && kt0 < p.k_tiles; kt0 += MX_SCALE_AHEAD) {
#pragma unroll
                for (int i = 0; i < MX_SCALE_AHEAD; ++i) {
                    const int kt = kt0 + i;
                    if (kt >= p.k_tiles) break;
                    const uint4 cur = q[i];
                    if (kt + MX_SCALE_AHEAD < p.k_tiles) q[i] = load_slice(kt + MX_SCALE_AHEAD);
                    if (!__all_sync(0xffffffffu, mx_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u, abort_flag))) { ok = false; break; }
                    *reinterpret_cast<uint4*>(tiles_ptr + stage * MX_STAGE_BYTES + G::SFX_OFF + lane * 16) = cur;
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ctl->full[stage]));
                    if (++stage == MX_STAGES) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == MX_COPY_WARP) {
        // ================= scale copies =================
        // Every ring stage has its own scale slot in tensor memory (as in the pair kernel): full[stage] can only complete
        // after the MMAs that read the slot's previous contents have.
        {
            uint32_t stage = 0, phase = 0;
            bool ok = true;
            for (long long t = blockIdx.x; ok && t < n_tiles_total; t += gridDim.x) {
                for (int kt = 0; kt < p.k_tiles; ++kt) {
                    if (!__all_sync(0xffffffffu, mx_wait(smem_u32(&ctl->full[stage]), phase, abort_flag))) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t sfw_t = tmem_base + G::SF_COL0 + stage * 8;
                    if (elect_one()) {
                        mx_copy_scales(sfw_t, mx_scale_desc(stage_base(stage) + G::SFW_OFF));
                        mx_copy_scales(sfw_t + 4, mx_scale_desc(stage_base(stage) + G::SFX_OFF));
                        tc_commit_local<false>(smem_u32(&ctl->sf_full[stage]));
                    }
                    __syncwarp();
                    if (++stage == MX_STAGES) { stage = 0; phase ^= 1u; }
                }
            }
            // all issued copies must have retired before tensor memory is released
            if (elect_one()) {
                tc_commit_local<false>(smem_u32(&ctl->drain_copy));
                const unsigned long long t0 = global_timer_ns();
                while (!mbar_try_wait(smem_u32(&ctl->drain_copy), 0) && global_timer_ns() - t0 < WAIT_LIMIT_NS) {}
            }
        }
        __syncwarp();
    } else {
        // ================= epilogue (warps 3..6) =================
        // A full block of 32 rows x 32 features goes through the warp's staging buffer and leaves as a bulk tensor store; of a
        // block that the expert only partly fills the rows are stored directly.
        //   not swapped  lane = row, tensor-memory column = feature: the warp has one slab of 32 rows and all features
        //   swapped      lane = feature, column = row: the warp has 32 features and all rows; the block is transposed on its
        //                way into the staging buffer (2-byte stores, 64 contiguous bytes per warp instruction)
        const int quarter = warp & 3;   // tensor-memory lanes [32 * quarter, 32 * quarter + 32)
        uint8_t* stage_ptr = tiles_ptr + MX_STAGES * MX_STAGE_BYTES + quarter * 2048;
        const int sw = (lane >> 1) & 3, piece = lane >> 3, within = (lane & 7) * 2;
        uint32_t n_stores = 0, acc = 0, acc_phase = 0;
        for (long long t = blockIdx.x; t < n_tiles_total; t += gridDim.x) {
            const MxTile tl = mx_decode<ROWS>(p, offs, tile_prefix, t);
            if (!__all_sync(0xffffffffu, mx_wait(smem_u32(&ctl->tmem_full[acc]), acc_phase, abort_flag))) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + acc * ROWS + ((uint32_t)(quarter * 32) << 16);
            const int n_rows = tl.row_end - tl.row0;
#pragma unroll 1
            for (int c = 0; c < ROWS / 32; ++c) {   // the warp's blocks
                const int r = (G::SWAPPED ? c : quarter) * 32, f = tl.n0 + (G::SWAPPED ? quarter : c) * 32;
                const int rv = min(32, n_rows - r);
                if (rv <= 0) break;
                uint32_t v[32];
                tc_ld32(taddr + c * 32, v);
                tc_wait_ld();
                if (rv == 32) {
                    if (n_stores != 0) {
                        if (lane == 0) bulk_wait_read0();
                        __syncwarp();
                    }
                    if (G::SWAPPED) {
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            *reinterpret_cast<__nv_bfloat16*>(stage_ptr + j * 64 + (((piece ^ ((j >> 1) & 3)) << 4) + within)) =
                                __float2bfloat16_rn(__uint_as_float(v[j]));
                    } else {
                        uint32_t w[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j) w[j] = pack_bf16(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            *reinterpret_cast<uint4*>(stage_ptr + lane * 64 + ((j ^ sw) << 4)) =
                                make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_2d(&map_o, f, tl.row0 + r, smem_u32(stage_ptr));
                        bulk_commit();
                    }
                    ++n_stores;
                } else if (G::SWAPPED) {
                    bf16* dst = p.out + ((long long)tl.row0 + r) * p.ldo + f + lane;
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j < rv) dst[(long long)j * p.ldo] = __float2bfloat16_rn(__uint_as_float(v[j]));
                } else if (lane < rv) {
                    uint4* d4 = reinterpret_cast<uint4*>(p.out + ((long long)tl.row0 + r + lane) * p.ldo + f);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        d4[j] = make_uint4(pack_bf16(__uint_as_float(v[8 * j]), __uint_as_float(v[8 * j + 1])),
                                           pack_bf16(__uint_as_float(v[8 * j + 2]), __uint_as_float(v[8 * j + 3])),
                                           pack_bf16(__uint_as_float(v[8 * j + 4]), __uint_as_float(v[8 * j + 5])),
                                           pack_bf16(__uint_as_float(v[8 * j + 6]), __uint_as_float(v[8 * j + 7])));
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl->tmem_empty[acc]));
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (n_stores != 0 && lane == 0) bulk_wait_all0();
        __syncwarp();
    }

    grid_launch_dependents();   // as late as this: see common.cuh
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)G::TMEM_COLS) : "memory");
    }
}

// ---- the CTA-pair form ----------------------------------------------------------------------------------
// Two CTAs of a cluster share one tile of M = 256, N up to 208 (tcgen05.mma.cta_group::2): each keeps 128 of the M side's codes
// and half of the N side's in shared memory, so a K slice of 128 costs each SM 29 KB of operand loads against 58 KB per two
// 128 x 128 tiles of the single-CTA form, which the L2 -> SM path bounds.  208, not 256: the two accumulators (tensor-memory
// columns 0 and 256) leave 48 columns behind each for three 16-column scale slots, one slot per ring stage.
//   weights on M       M side: 256 output features of an expert's weights.  N side: its rows, in equal tiles of at most 208 rows
//                      (a multiple of 16), so that almost no tensor work goes to padding.  The accumulator has a feature per
//                      lane and a row per column and is transposed on its way out.
//   rows on M          M side: 256 rows of an expert, half a tile of padding on average.  N side: 208 features (the last tile is narrower).
//   weight gradients   M side: 256 rows of the output, N side: 208 columns of it (the last tile is narrower).
// Rows on M against weights on M: all four GEMMs
// 18 % faster at 384 rows per expert (64 experts of 2048 x 1408: gate/up 206 -> 166, down 108 -> 88 us), 3-8 % at 1024
// (128 of 2048 x 768: 433 -> 402, 282 -> 272 us), 3-6 % at 2048 (8 of 4096 x 14336: 1697 -> 1649, 884 -> 827 us), 10 % under
// Dirichlet loads (128 of 2944 x 2944).  Not where it has the more tiles: mx_form.
//   scale factors: each CTA holds the scales of its own 128 of the M side (4 columns) and of ALL the tile's N side (two blocks of
//   128, 8 columns) in its own tensor memory; tcgen05.cp.cta_group::2, issued once, copies in both CTAs from the same
//   shared-memory offsets.  Weight-scale blocks (on M: 512 bytes per 128 features and K slice, on N: 1024 bytes per 208) and the
//   weight gradients' N-side blocks (1024 bytes per 208 columns) are contiguous in global memory and arrive by one tensor copy;
//   scales of packed rows are gathered by a warp.
//   warp 0      TMA producer (both CTAs; all loads complete on the first CTA's full[stage], as in the bf16 pair kernels)
//   warp 1      first CTA: issues the MMAs and the commits for the pair
//   warp 2      scales of packed rows (weights on M: the N side's) or of the M side's 128 rows
//   warps 3..10 epilogue: a 32-lane quarter x every other 32-column block
//   warp 11     first CTA: issues the scale copies (smem -> tensor memory) of each stage
// What bounds it: a K slice takes ~590 cycles where the tensor pipe needs ~420 (four N = 208 MMAs): operand reads by the tensor
// core and fills by the TMA unit together ask shared memory for ~140 bytes per cycle at this tile width (halving the waits and
// commits per slice changed nothing; with scale copies in the MMA thread it took ~770, with two or four scale slots ~510 before
// a load was issued).  The largest shapes run into the power cap.
constexpr int MXP_NT = 208;                 // most of a tile's N over the pair
constexpr int MXP_ROWS = 2 * MX_BM;         // a tile's M over the pair
constexpr int MXP_STAGES = 6;
constexpr int MXP_A_BYTES = MX_BM * MX_BK;              // 16 KB
constexpr int MXP_B_BYTES = (MXP_NT / 2) * MX_BK;       // 13 KB
constexpr int MXP_SFA_OFF = MXP_A_BYTES + MXP_B_BYTES;  // 512 bytes: scales of this CTA's part of the M side
constexpr int MXP_SFB_OFF = MXP_SFA_OFF + 512;          // 1024 bytes: scales of the tile's N side
constexpr int MXP_STAGE_BYTES = 31 * 1024;              // 30.5 KB used; stages stay 1024-byte aligned
constexpr int MXP_LOW_BOX = 64;                         // weights on M: rows of the smaller of the two boxes of row codes
constexpr int MXP_EPI_WARPS = 8;
constexpr int MXP_COPY_WARP = 3 + MXP_EPI_WARPS;   // the scale-copy warp comes after the epilogue warps
constexpr int MXP_THREADS = 32 * (4 + MXP_EPI_WARPS);
constexpr int MXP_STAGING_BYTES = MXP_EPI_WARPS * 2048;
constexpr int MXP_ACC_STRIDE = 256;         // tensor-memory columns between the two accumulators
// one scale slot (16 columns) per ring stage, three behind each accumulator: a stage's slot is free when the stage is
__device__ __forceinline__ uint32_t mxp_slot_col(uint32_t stage) { return MXP_NT + (stage / 3u) * MXP_ACC_STRIDE + (stage % 3u) * 16; }
static_assert(MXP_STAGES == 6 && MXP_NT + 3 * 16 <= MXP_ACC_STRIDE, "scale slots");
static_assert(MXP_SFB_OFF + 1024 <= MXP_STAGE_BYTES, "stage layout");

struct MxPairCtl {
    unsigned long long full[MXP_STAGES];
    unsigned long long sf_full[MXP_STAGES];   // first CTA: the stage's scales are in tensor memory (and its operands landed)
    unsigned long long empty[MXP_STAGES];
    unsigned long long tmem_full[2];
    unsigned long long tmem_empty[2];
    unsigned long long drain;
    unsigned long long drain_copy;
    uint32_t tmem_base;
    int abort_flag;
    int stage_n[MXP_STAGES];   // N of the tile a stage belongs to (published by the first CTA's producer)
    int32_t offs[MX_MAX_E + 1];          // row-ragged forms: offsets; weight gradients: slice_prefix
    int32_t tile_prefix[MX_MAX_E + 1];   // row-ragged forms: row tiles of the experts before e
};
constexpr int MXP_SMEM_BYTES = MXP_STAGES * MXP_STAGE_BYTES + MXP_STAGING_BYTES + 1024 + (int)sizeof(MxPairCtl);
static_assert(MXP_SMEM_BYTES <= 232448, "exceeds the shared memory a CTA can opt in to");

// The pair kernel serves two problems, the first in two forms (template parameter FORM):
//   row-ragged GEMM   out[r, :] = a[r, :] . b[e]^T for the rows r of expert e: row tiles from `offsets`, the
//                     contraction is k_tiles slices for every tile, b and its scale blocks are indexed by expert;
//   weight gradient   dW[e] [M, N] = A_e^T B_e with token-quantised, transposed operands (further down): a fixed tile
//                     list (expert x M tiles x N tiles), the contraction of expert e is the slices
//                     [slice_prefix[e], slice_prefix[e + 1]) of both operands, nothing is indexed by expert but the output.
struct MxPairParams {
    const int32_t* prefix;   // offsets [E + 1] / slice_prefix [E + 1]
    int E, k_tiles, n_tiles, m_tiles, n_cols, n_slices;   // k_tiles: row-ragged forms; m_tiles, n_slices: weight gradients
    int M;                   // weight gradients: rows of one expert's output
    long long sa_rows;       // words per slice of `sa`: R / M
    const uint32_t* sa;      // scale words of the packed rows / of the A side [slices][sa_rows]
    bf16* out;
    long long ldo;
};

__device__ __forceinline__ uint32_t mxp_idesc(uint32_t n, uint32_t sf) {
    return (sf << 4) | ((n >> 3) << 17) | (1u << 23) | ((uint32_t)(MXP_ROWS >> 4) << 24) | (sf << 29);
}
__device__ __forceinline__ void mxp_copy_scales(uint32_t taddr, uint64_t sdesc) {
    asm volatile("tcgen05.cp.cta_group::2.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}
__device__ __forceinline__ void mxp_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t sfa,
                                        uint32_t sfb, uint32_t accumulate) {
    asm volatile(
        "{ .reg .pred p; setp.ne.u32 p, %4, 0;"
        " tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale [%0], %1, %2, %3, [%5], [%6], p; }" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb)
        : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t v[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}

enum MxPairForm { MXP_WEIGHTS_M = 0, MXP_ROWS_M = 1, MXP_WGRAD = 2 };
struct MxPairTile {
    int row0;               // weight gradients: first output row inside the expert's output; row-ragged forms: first packed row
    int rows;               // rows from there to the end of the expert's output; row-ragged forms: of the expert, at most a tile's
    int out_row0;           // weight gradients: first row of the expert's output in the output tensor
    int n0, width;          // first output column (feature); N of the MMAs
    int k0, k_tiles;        // K slices [k0, k0 + k_tiles) of both operands
    int w_row, sf_row0;     // first row of the tile in the B codes (weight gradients) / weight codes; row of its first scale block
};
template <int FORM>
__device__ __forceinline__ MxPairTile mxp_decode(const MxPairParams& p, const MxPairCtl* ctl, long long t) {
    MxPairTile tl;
    if (FORM == MXP_WGRAD) {
        const int per_e = p.m_tiles * p.n_tiles;
        const int e = (int)(t / per_e);
        const int local = (int)(t - (long long)e * per_e);
        const int nt = local / p.m_tiles;   // column tile major inside an expert: the pairs running together share the B tile in L2
        tl.row0 = (local - nt * p.m_tiles) * MXP_ROWS;
        tl.rows = p.M - tl.row0;
        tl.out_row0 = e * p.M;
        tl.k0 = ctl->offs[e];
        tl.k_tiles = ctl->offs[e + 1] - tl.k0;
        tl.n0 = nt * MXP_NT;
        tl.width = min(MXP_NT, p.n_cols - tl.n0);
        tl.w_row = tl.n0;
        tl.sf_row0 = nt * p.n_slices + tl.k0;
    } else {
        int lo = 0, hi = p.E;   // largest e with tile_prefix[e] * n_tiles <= t
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if ((long long)ctl->tile_prefix[mid] * p.n_tiles <= t) lo = mid; else hi = mid;
        }
        const int local = (int)(t - (long long)ctl->tile_prefix[lo] * p.n_tiles);
        const int m_tiles_e = ctl->tile_prefix[lo + 1] - ctl->tile_prefix[lo];
        const int nt = local / m_tiles_e, mt = local - nt * m_tiles_e;   // feature tile major inside an expert (the pairs running together share weight tiles in L2)
        const int n_e = ctl->offs[lo + 1] - ctl->offs[lo];
        // rows on the N side: equal tiles, the last one takes what is left
        const int per_tile = FORM == MXP_ROWS_M ? MXP_ROWS : ((n_e + m_tiles_e - 1) / m_tiles_e + 15) & ~15;
        tl.row0 = ctl->offs[lo] + mt * per_tile;
        tl.rows = min(per_tile, ctl->offs[lo + 1] - tl.row0);
        tl.out_row0 = 0;
        tl.k0 = 0;
        tl.k_tiles = p.k_tiles;
        tl.n0 = nt * (FORM == MXP_ROWS_M ? MXP_NT : MXP_ROWS);
        tl.width = FORM == MXP_ROWS_M ? min(MXP_NT, p.n_cols - tl.n0) : (tl.rows + 15) & ~15;
        tl.w_row = lo * p.n_cols + tl.n0;
        tl.sf_row0 = (FORM == MXP_ROWS_M ? lo * p.n_tiles + nt : lo * (p.n_cols >> 7) + 2 * nt) * p.k_tiles;
    }
    return tl;
}
// K slices of tile t (the roles that do not need the rest of the tile)
template <int FORM>
__device__ __forceinline__ int mxp_k_tiles(const MxPairParams& p, const MxPairCtl* ctl, long long t) {
    if (FORM != MXP_WGRAD) return p.k_tiles;
    const int e = (int)(t / ((long long)p.m_tiles * p.n_tiles));
    return ctl->offs[e + 1] - ctl->offs[e];
}

template <int FORM>
__global__ void __launch_bounds__(MXP_THREADS, 1)
mx_pair_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                    const __grid_constant__ CUtensorMap map_b_low, const __grid_constant__ CUtensorMap map_sf,
                    const __grid_constant__ CUtensorMap map_o, const MxPairParams p) {
    constexpr bool ROWS_N = FORM == MXP_WEIGHTS_M;   // the packed rows are the N side
    extern __shared__ uint8_t smem_raw[];
    const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* tiles_ptr = smem_raw + (tiles_base - smem_u32(smem_raw));
    MxPairCtl* ctl = reinterpret_cast<MxPairCtl*>(tiles_ptr + MXP_STAGES * MXP_STAGE_BYTES + MXP_STAGING_BYTES);
    volatile int* abort_flag = &ctl->abort_flag;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (uniform, and known to be)
    const uint32_t rank = cluster_ctarank();   // 0 = the CTA that issues the MMAs
    const long long first_tile = blockIdx.x >> 1, tile_stride = gridDim.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < MXP_STAGES; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 4);   // per CTA: the producer's arrive (with its byte count) + the scale warp's
            mbar_init(smem_u32(&ctl->sf_full[s]), 1);
            mbar_init(smem_u32(&ctl->empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(&ctl->tmem_full[a]), 1);
            mbar_init(smem_u32(&ctl->tmem_empty[a]), 2 * MXP_EPI_WARPS);
        }
        mbar_init(smem_u32(&ctl->drain), 1);
        mbar_init(smem_u32(&ctl->drain_copy), 1);
        ctl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_tmap(&map_a);
        prefetch_tmap(&map_b);
        prefetch_tmap(&map_b_low);
        prefetch_tmap(&map_sf);
        prefetch_tmap(&map_o);
    }
    // everything above may run while the kernel before is still finishing; the schedule is derived from its output
    grid_dependency_wait();
    for (int e = threadIdx.x; e <= p.E; e += MXP_THREADS) ctl->offs[e] = p.prefix[e];
    __syncthreads();
    if (FORM != MXP_WGRAD && warp == 0) exclusive_tile_prefix(ctl->offs, ctl->tile_prefix, p.E, ROWS_N ? MXP_NT : MXP_ROWS, lane);
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                     "r"((uint32_t)MX_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();   // the other CTA's barriers and tensor memory exist from here on
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, ctl->tmem_base, 0);
    const long long n_tiles_total = FORM == MXP_WGRAD ? (long long)p.E * p.m_tiles * p.n_tiles : (long long)__shfl_sync(0xffffffffu, ctl->tile_prefix[p.E], 0) * p.n_tiles;
    const uint32_t full0 = map_to_cta(smem_u32(&ctl->full[0]), 0);   // full[] of the MMA-issuing CTA

    if (warp == 0) {
        // ================= producer (both CTAs; each fills its own ring) =================
        {   // the whole warp on uniform values, one elected lane issues (see the bf16 kernels)
            uint32_t stage = 0, phase = 0, issued = 0;
            bool ok = true;
            for (long long t = first_tile; ok && t < n_tiles_total; t += tile_stride) {
                MxPairTile tl = mxp_decode<FORM>(p, ctl, t);
                auto uni = [](int v) { return __shfl_sync(0xffffffffu, v, 0); };
                tl.row0 = uni(tl.row0); tl.width = uni(tl.width); tl.k0 = uni(tl.k0); tl.k_tiles = uni(tl.k_tiles); tl.w_row = uni(tl.w_row);
                // this CTA's 128 rows of the M side, its half of the N side, its scale blocks
                const int my_n = tl.width >> 1;
                const int a_row = (ROWS_N ? tl.w_row : tl.row0) + (int)rank * MX_BM, b_row = (ROWS_N ? tl.row0 : tl.w_row) + (int)rank * my_n;
                const int sf_row0 = uni(tl.sf_row0) + (ROWS_N ? (int)rank * tl.k_tiles : 0);
                const bool low = ROWS_N && my_n <= MXP_LOW_BOX;
                const uint32_t bytes = ROWS_N ? MXP_A_BYTES + (low ? MXP_LOW_BOX * MX_BK : MXP_B_BYTES) + 512 : MXP_A_BYTES + MXP_B_BYTES + 1024;
                for (int kt = 0; kt < tl.k_tiles; ++kt) {
                    if (!__all_sync(0xffffffffu, mx_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u, abort_flag))) { ok = false; break; }
#ifdef MOE_TEST_HOOKS
                    if (g_mx_test_withhold_first_stage != 0 && issued == 0) {
                        ++issued;
                        if (++stage == MXP_STAGES) { stage = 0; phase ^= 1u; }
                        continue;
                    }
#endif
                    if (elect_one()) {
                        if (rank == 0) ctl->stage_n[stage] = tl.width;   // read by the MMA thread after its wait on full[stage]
                        const uint32_t bar = full0 + stage * (uint32_t)sizeof(unsigned long long);
                        const uint32_t dst = tiles_base + stage * MXP_STAGE_BYTES;
                        mbar_arrive_expect_tx_cluster(bar, bytes);
                        tma_load_2d_pair(dst, &map_a, (tl.k0 + kt) * MX_BK, a_row, bar);
                        tma_load_2d_pair(dst + MXP_A_BYTES, low ? &map_b_low : &map_b, (tl.k0 + kt) * MX_BK, b_row, bar);
                        tma_load_2d_pair(dst + (ROWS_N ? MXP_SFA_OFF : MXP_SFB_OFF), &map_sf, 0, sf_row0 + kt, bar);
                    }
                    __syncwarp();
                    ++issued;
                    if (++stage == MXP_STAGES) { stage = 0; phase ^= 1u; }
                }
            }
            if (!ok && issued != 0) {
                // leave no bulk copy in flight: the copies report to a barrier this thread cannot always poll (the other
                // CTA's), so outwait them -- a copy that was issued completes within microseconds
                const unsigned long long t0 = global_timer_ns();
                while (global_timer_ns() - t0 < 2000000ull) {}
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer: the first CTA's warp 1 =================
        // This warp, the producer and the scale-copy warp run whole, on warp-uniform values that the compiler knows to be
        // uniform, and one elected lane issues.  Loops under `if (lane == 0)` in the two others, with role index and tile
        // fields taken from vector registers, were 6-9 % slower: 8 large experts gate/up 1469 -> 1390 us (2.77 PFLOP/s),
        // 128 experts of width 768 397 -> 369 us, their weight gradient 203 -> 190 us.
        if (rank == 0) {
            uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0, n = MXP_NT;
            bool ok = true;
            for (long long t = first_tile; ok && t < n_tiles_total; t += tile_stride) {
                const int k_tiles_t = __shfl_sync(0xffffffffu, mxp_k_tiles<FORM>(p, ctl, t), 0);
                if (k_tiles_t == 0) continue;   // (weight gradients) an expert without rows: the epilogue writes zeros on its own
                if (!__all_sync(0xffffffffu, mx_wait(smem_u32(&ctl->tmem_empty[acc]), acc_phase ^ 1u, abort_flag))) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * MXP_ACC_STRIDE;
                for (int kt = 0; kt < k_tiles_t; ++kt) {
                    if (!__all_sync(0xffffffffu, mx_wait(smem_u32(&ctl->sf_full[stage]), phase, abort_flag))) { ok = false; break; }
                    tc_fence_after();
                    if (kt == 0) n = (uint32_t)__shfl_sync(0xffffffffu, ctl->stage_n[stage], 0);
                    const uint32_t s_base = tiles_base + stage * MXP_STAGE_BYTES;
                    const uint32_t sfa_t = tmem_base + mxp_slot_col(stage), sfb_t = sfa_t + 4;
                    const uint64_t a_desc = mx_operand_desc(s_base), b_desc = mx_operand_desc(s_base + MXP_A_BYTES);
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < MX_BK / 32; ++k)
                            mxp_mma(d_tmem, a_desc + (uint64_t)((k * 32) >> 4), b_desc + (uint64_t)((k * 32) >> 4), mxp_idesc(n, k),
                                    sfa_t, sfb_t, (kt != 0 || k != 0) ? 1u : 0u);
                        tc_commit<true>(smem_u32(&ctl->empty[stage]));
                    }
                    __syncwarp();
                    if (++stage == MXP_STAGES) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                if (elect_one()) tc_commit<true>(smem_u32(&ctl->tmem_full[acc]));
                __syncwarp();
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
            // all issued MMAs must have retired before tensor memory is released
            if (elect_one()) {
                tc_commit_local<true>(smem_u32(&ctl->drain));
                const unsigned long long t0 = global_timer_ns();
                while (!mbar_try_wait(smem_u32(&ctl->drain), 0) && global_timer_ns() - t0 < WAIT_LIMIT_NS) {}
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // ================= scales of the rows =================
        // On the M side: this CTA's 128 rows.  On the N side: all the tile's rows in both CTAs
        // (at most 208: seven words per lane and slice, two blocks of 128 rows; columns past the tile's N are never read).
        constexpr int WORDS = ROWS_N ? 7 : 4;
        uint32_t stage = 0, phase = 0;
        bool ok = true;
        for (long long t = first_tile; ok && t < n_tiles_total; t += tile_stride) {
            const MxPairTile tl = mxp_decode<FORM>(p, ctl, t);
            long long rows[WORDS];
#pragma unroll
            for (int i = 0; i < WORDS; ++i) {
                const long long r = (long long)tl.row0 + (ROWS_N ? 0 : (int)rank * MX_BM) + 32 * i + lane;
                rows[i] = r < p.sa_rows ? r : p.sa_rows - 1;   // rows past the end are never stored; any valid address will do
            }
            // the words of MX_SCALE_AHEAD slices are in flight at any time: one slice per global-load round trip would
            // bound the whole pipeline (the loads wait behind the operand traffic)
            struct Words { uint32_t w[8]; };
            auto load_slice = [&](int kt) {
                const uint32_t* s = p.sa + (long long)(tl.k0 + kt) * p.sa_rows;
                Words q;
#pragma unroll
                for (int i = 0; i < 8; ++i) q.w[i] = i < WORDS ? __ldg(s + rows[i < WORDS ? i : 0]) : 0u;
                return q;
            };
            Words q[MX_SCALE_AHEAD];
#pragma unroll
            for (int i = 0; i < MX_SCALE_AHEAD; ++i) q[i] = load_slice(min(i, max(tl.k_tiles - 1, 0)));
            for (int kt0 = 0; ok && kt0 < tl.k_tiles; kt0 += MX_SCALE_AHEAD) {
#pragma unroll
                for (int i = 0; i < MX_SCALE_AHEAD; ++i) {
                    const int kt = kt0 + i;
                    if (kt >= tl.k_tiles) break;
                    const Words cur = q[i];
                    if (kt + MX_SCALE_AHEAD < tl.k_tiles) q[i] = load_slice(kt + MX_SCALE_AHEAD);
                    if (!__all_sync(0xffffffffu, mx_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u, abort_flag))) { ok = false; break; }
                    uint8_t* to = tiles_ptr + stage * MXP_STAGE_BYTES + (ROWS_N ? MXP_SFB_OFF : MXP_SFA_OFF) + lane * 16;
                    *reinterpret_cast<uint4*>(to) = make_uint4(cur.w[0], cur.w[1], cur.w[2], cur.w[3]);
                    if (ROWS_N) *reinterpret_cast<uint4*>(to + 512) = make_uint4(cur.w[4], cur.w[5], cur.w[6], cur.w[7]);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive_remote(full0 + stage * (uint32_t)sizeof(unsigned long long));
                    if (++stage == MXP_STAGES) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == MXP_COPY_WARP) {
        // ================= scale copies: first CTA =================
        // Takes the three tcgen05.cp per K slice off the MMA thread (each tcgen05 instruction costs the issuing thread
        // 60-85 cycles; with them the MMA thread needed ~770 cycles per slice).  Every ring stage has its own scale slot in
        // tensor memory: full[stage] can only complete after the stage was released, i.e. after the MMAs that read the
        // slot's previous contents have completed.
        if (rank == 0) {
            uint32_t stage = 0, phase = 0;
            bool ok = true;
            for (long long t = first_tile; ok && t < n_tiles_total; t += tile_stride) {
                const int k_tiles_t = __shfl_sync(0xffffffffu, mxp_k_tiles<FORM>(p, ctl, t), 0);
                for (int kt = 0; kt < k_tiles_t; ++kt) {
                    if (!__all_sync(0xffffffffu, mx_wait(smem_u32(&ctl->full[stage]), phase, abort_flag))) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t s_base = tiles_base + stage * MXP_STAGE_BYTES;
                    const uint32_t sfa_t = tmem_base + mxp_slot_col(stage), sfb_t = sfa_t + 4;
                    if (elect_one()) {
                        mxp_copy_scales(sfa_t, mx_scale_desc(s_base + MXP_SFA_OFF));
                        mxp_copy_scales(sfb_t, mx_scale_desc(s_base + MXP_SFB_OFF));
                        mxp_copy_scales(sfb_t + 4, mx_scale_desc(s_base + MXP_SFB_OFF + 512));
                        tc_commit_local<true>(smem_u32(&ctl->sf_full[stage]));
                    }
                    __syncwarp();
                    if (++stage == MXP_STAGES) { stage = 0; phase ^= 1u; }
                }
            }
            // all issued copies must have retired before tensor memory is released
            if (elect_one()) {
                tc_commit_local<true>(smem_u32(&ctl->drain_copy));
                const unsigned long long t0 = global_timer_ns();
                while (!mbar_try_wait(smem_u32(&ctl->drain_copy), 0) && global_timer_ns() - t0 < WAIT_LIMIT_NS) {}
            }
        }
        __syncwarp();
    } else {
        // ================= epilogue (warps 3..10, both CTAs) =================
        const int quarter = warp & 3;          // tensor-memory lanes [32 * quarter, 32 * quarter + 32)
        const int half = (warp - 3) >> 2;      // 32-column blocks 0, 2, 4, 6 or 1, 3, 5 (+ the 16-column tail)
        uint8_t* stage_ptr = tiles_ptr + MXP_STAGES * MXP_STAGE_BYTES + (warp - 3) * 2048;
        const int sw = (lane >> 1) & 3;
        const uint32_t empty0 = map_to_cta(smem_u32(&ctl->tmem_empty[0]), 0);
        uint32_t n_stores = 0, acc = 0, acc_phase = 0;
        for (long long t = first_tile; t < n_tiles_total; t += tile_stride) {
            const MxPairTile tl = mxp_decode<FORM>(p, ctl, t);
            const bool have_acc = tl.k_tiles != 0;
            if (have_acc) {
                if (!__all_sync(0xffffffffu, mx_wait(smem_u32(&ctl->tmem_full[acc]), acc_phase, abort_flag))) break;
                tc_fence_after();
            }
            const uint32_t taddr = tmem_base + acc * MXP_ACC_STRIDE + ((uint32_t)(quarter * 32) << 16);
            if (ROWS_N) {
                // lane = feature, column = row: the two warps of a lane quarter take the 32-row blocks alternately; a block is
                // transposed on its way into the staging buffer
                const int f = tl.n0 + (int)rank * MX_BM + quarter * 32;
#pragma unroll 1
                for (int c = half; f < p.n_cols && c * 32 < tl.rows; c += 2) {
                    uint32_t v[32], w[16];
                    tc_ld_frag32(taddr + c * 32, v);
                    tc_wait_ld();
                    const int r0 = tl.row0 + c * 32, rv = min(32, tl.rows - c * 32);
                    pack_frag(v, w);
                    if (n_stores != 0) {
                        if (lane == 0) bulk_wait_read0();
                        __syncwarp();
                    }
                    store_frag(smem_u32(stage_ptr) + frag_offset(lane), w);
                    if (rv == 32) {
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) {
                            tma_store_2d(&map_o, f, r0, smem_u32(stage_ptr));
                            bulk_commit();
                        }
                        ++n_stores;
                    } else {
                        __syncwarp();
                        copy_block_rows(stage_ptr, p.out + (long long)r0 * p.ldo + f, p.ldo, rv, lane);
                        __syncwarp();
                    }
                }
            }
            const int slab_in = (int)rank * MX_BM + quarter * 32;   // first row of this warp's slab, inside the tile
            const int rows_valid = max(0, min(32, tl.rows - slab_in));
            const int slab0 = tl.out_row0 + tl.row0 + slab_in;      // ... and in the output tensor
#pragma unroll 1
            for (int c = half; !ROWS_N && c < 8; c += 2) {
                const int left = tl.width - 32 * c;   // columns of the tile from this block on (warp-uniform)
                if (left <= 0) break;
                const int n = tl.n0 + c * 32;
                uint32_t w[16];
                if (!have_acc) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) w[j] = 0u;
                } else if (left >= 32) {
                    uint32_t v[32];
                    tc_ld32(taddr + c * 32, v);
                    tc_wait_ld();
#pragma unroll
                    for (int j = 0; j < 16; ++j) w[j] = pack_bf16(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
                } else {
                    uint32_t v[16];
                    tc_ld16(taddr + c * 32, v);
                    tc_wait_ld();
#pragma unroll
                    for (int j = 0; j < 8; ++j) w[j] = pack_bf16(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
                }
                if (rows_valid == 0) continue;
                if (left >= 32 && rows_valid == 32) {
                    if (n_stores != 0) {
                        if (lane == 0) bulk_wait_read0();
                        __syncwarp();
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        *reinterpret_cast<uint4*>(stage_ptr + lane * 64 + ((j ^ sw) << 4)) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_2d(&map_o, n, slab0, smem_u32(stage_ptr));
                        bulk_commit();
                    }
                    ++n_stores;
                } else if (lane < rows_valid) {
                    uint4* d4 = reinterpret_cast<uint4*>(p.out + ((long long)slab0 + lane) * p.ldo + n);
                    d4[0] = make_uint4(w[0], w[1], w[2], w[3]);
                    d4[1] = make_uint4(w[4], w[5], w[6], w[7]);
                    if (left >= 32) {
                        d4[2] = make_uint4(w[8], w[9], w[10], w[11]);
                        d4[3] = make_uint4(w[12], w[13], w[14], w[15]);
                    }
                }
            }
            if (!have_acc) continue;
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(empty0 + acc * (uint32_t)sizeof(unsigned long long));
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (n_stores != 0 && lane == 0) bulk_wait_all0();
        __syncwarp();
    }

    grid_launch_dependents();   // as late as this: see common.cuh
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();   // neither CTA's shared memory / barriers may go away while the other still uses them
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)MX_TMEM_COLS) : "memory");
    }
}

// ---- quantisers ---------------------------------------------------------------------------------------
// scale exponent of a block with largest magnitude amax: floor(log2 amax) - 8, clamped to the E8M0 range; -127 for zero
__device__ __forceinline__ int mx_scale_exp(float amax) {
    if (!(amax > 0.f)) return -127;
    const int field = (__float_as_int(amax) >> 23) & 0xFF;             // amax is positive and finite
    const int e = (field != 0 ? field - 127 : ilogbf(amax)) - 8;       // subnormal magnitudes take the library route
    return e < -127 ? -127 : (e > 127 ? 127 : e);
}
// 2^-s as a float (s in [-127, 127]; 2^-127 is a subnormal)
__device__ __forceinline__ float mx_inv_scale(int s) {
    return s == 127 ? __int_as_float(0x00400000) : __int_as_float((127 - s) << 23);
}
// two values -> two codes (the first in the low byte), one conversion instruction
__device__ __forceinline__ uint32_t mx_e4m3x2(float lo, float hi) {
    return (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(lo, hi), __NV_SATFINITE, __NV_E4M3);
}

// Largest magnitude of the 8 bf16 values of a 16-byte piece, kept packed (two running maxima, one per half word).  The
// maximum of bf16 values is exact, so the packed form decides the same scale as the fp32 one; a NaN loses against any number.
__device__ __forceinline__ __nv_bfloat162 mx_max2(uint32_t a, uint32_t b) {
    return __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
}
__device__ __forceinline__ uint32_t mx_abs_max4(const uint4& v) {
    const __nv_bfloat162 m = __hmax2(mx_max2(v.x & 0x7fff7fffu, v.y & 0x7fff7fffu), mx_max2(v.z & 0x7fff7fffu, v.w & 0x7fff7fffu));
    return *reinterpret_cast<const uint32_t*>(&m);
}
__device__ __forceinline__ uint32_t mx_abs_max(uint32_t a, uint32_t b) {   // of packed magnitudes
    const __nv_bfloat162 m = mx_max2(a, b);
    return *reinterpret_cast<const uint32_t*>(&m);
}
__device__ __forceinline__ float mx_lo(uint32_t w) { return __uint_as_float(w << 16); }          // bf16 -> fp32 is a shift
__device__ __forceinline__ float mx_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
// 2^-s as bf16 bits (exact: it is a power of two), and its product with two packed values: exact but for results so small
// that their code is zero, so the codes are those of the fp32 product at half the multiplications.
__device__ __forceinline__ uint32_t mx_inv_bits(int s) { return (uint32_t)__float_as_int(mx_inv_scale(s)) >> 16; }
__device__ __forceinline__ uint32_t mx_scale2(uint32_t v, uint32_t inv2) {
    const __nv_bfloat162 m = __hmul2(*reinterpret_cast<const __nv_bfloat162*>(&v), *reinterpret_cast<const __nv_bfloat162*>(&inv2));
    return *reinterpret_cast<const uint32_t*>(&m);
}
__device__ __forceinline__ uint2 mx_codes8(const uint4& v, int se) {   // 8 consecutive values -> 8 code bytes
    const uint32_t inv = mx_inv_bits(se), inv2 = inv | (inv << 16);
    const uint32_t x = mx_scale2(v.x, inv2), y = mx_scale2(v.y, inv2), z = mx_scale2(v.z, inv2), w = mx_scale2(v.w, inv2);
    return make_uint2(mx_e4m3x2(mx_lo(x), mx_hi(x)) | (mx_e4m3x2(mx_lo(y), mx_hi(y)) << 16),
                      mx_e4m3x2(mx_lo(z), mx_hi(z)) | (mx_e4m3x2(mx_lo(w), mx_hi(w)) << 16));
}
// Scale exponent of a block of 32 values held by 4 consecutive lanes, 8 each.
__device__ __forceinline__ int mx_block_exp(const uint4& v) {
    uint32_t m = mx_abs_max4(v);
    m = mx_abs_max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = mx_abs_max(m, __shfl_xor_sync(0xffffffffu, m, 2));
    return mx_scale_exp(fmaxf(mx_lo(m), mx_hi(m)));
}
// 32 bytes (16 bf16 values) with one load if the operand is 32-byte aligned, as two halves if only 16 (what callers owe).
__device__ __forceinline__ void mx_load32(const uint4* p, bool whole, uint4& lo, uint4& hi) {
    if (whole) {
        asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(lo.x), "=r"(lo.y), "=r"(lo.z), "=r"(lo.w), "=r"(hi.x), "=r"(hi.y), "=r"(hi.z), "=r"(hi.w)
                     : "l"(p));
    } else {
        lo = __ldg(p);
        hi = __ldg(p + 1);
    }
}
// Scale exponent of a block of 32 values held by 2 consecutive lanes, 16 each.
__device__ __forceinline__ int mx_block_exp2(const uint4& lo, const uint4& hi) {
    uint32_t m = mx_abs_max(mx_abs_max4(lo), mx_abs_max4(hi));
    m = mx_abs_max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    return mx_scale_exp(fmaxf(mx_lo(m), mx_hi(m)));
}
__device__ __forceinline__ uint4 mx_codes16(const uint4& lo, const uint4& hi, int se) {   // 16 consecutive values -> 16 code bytes
    const uint2 a = mx_codes8(lo, se), b = mx_codes8(hi, se);
    return make_uint4(a.x, a.y, b.x, b.y);
}
// Where the scale word of feature `f` (4 scale bytes of one K slice) sits inside a 128-feature block of 512 bytes, in words.
__device__ __forceinline__ int mx_sf_word(int f) { return (f % 32) * 4 + (f % 128) / 32; }
// The scale words of 128 features f0 .. f0 + 127 (f0 a multiple of 128) of one K slice, in shared memory, into both
// weight-scale tilings; `block` is the slice's 512-byte block of the first, `pair` the slice's place in the second
// (which the column tile's index times `pair_stride` is added to).  Threads 0..127.
__device__ __forceinline__ void mx_store_weight_scales(const uint32_t* words, int f0, uint32_t* block, uint8_t* pair, long long pair_stride,
                                                       int i) {
    if (block != nullptr) block[i] = words[(i % 4) * 32 + i / 4];   // consecutive threads, consecutive words
    const int nt = (f0 + i) / MXP_NT, c = (f0 + i) % MXP_NT;
    *reinterpret_cast<uint32_t*>(pair + nt * pair_stride + (c >> 7) * 512 + mx_sf_word(c) * 4) = words[i];
}

// rows x n bf16 -> codes (same layout) and scales.  A block takes 128 rows x one 128-wide slice; eight lanes hold a row (16
// elements per lane, one 32-byte load), four rows one after the other with their loads all in flight; the 2 lanes of a
// block of 32 agree on its scale through one shuffle.  The scale bytes meet in shared memory and leave as one 32-bit word
// per (row, slice):
//   WEIGHTS = false (activations): word [slice][row], 512 contiguous bytes per block of threads;
//   WEIGHTS = true  (weights whose contraction axis is contiguous, rows = E * n_feat, e.g. W_down read as [I, H] for the
//                    data gradient): the word's place in each of the two weight-scale tilings.  The output may be a
//                    column range of a wider operand (out_k_tiles slices per row, this input filling slices
//                    out_kt0 .. out_kt0 + n/128): W_gate and W_up side by side along the contraction of the gate/up
//                    data gradient.
// 3 bytes of HBM traffic per element, so bound by HBM only if few instructions and few partial sectors go into one.  201 M weights
// (128 x 768 x 2048) 115 -> 95 us (6.4 TB/s), two of them side by side 238 -> 194 us, activations 131072 x 2048 125 -> 122 us
// (6.6 TB/s), each against a half-warp per row with 16-byte loads and 8-byte stores.  (With a warp walking along a row, every
// (row, slice) took a 64-bit division, eight shuffles and, for weights, two 4-byte stores into a sector each: 242 and 184 us.)
template <bool WEIGHTS>
__global__ void __launch_bounds__(256) mx_quantize_rows_kernel(const uint4* __restrict__ x, long long rows, int n, int n_feat,
                                                               int out_k_tiles, int out_kt0, uint4* __restrict__ codes,
                                                               uint8_t* __restrict__ scales, uint8_t* __restrict__ scales_pair) {
    __shared__ __align__(16) uint8_t sf[128 * 4];
    if (!grid_dependency_wait_tested()) return;
    grid_launch_dependents();
    const int k_tiles = n >> 7;
    const int row_tile = (int)(blockIdx.x / (unsigned)k_tiles), kt = (int)(blockIdx.x - (unsigned)row_tile * (unsigned)k_tiles);
    const long long row0 = 128ll * row_tile;
    const int sub = threadIdx.x >> 3, l8 = threadIdx.x & 7;
    const int n_rows = (int)min(128ll, rows - row0);
    const bool whole = (reinterpret_cast<uintptr_t>(x) & 31) == 0;
    const uint4* src = x + (row0 + sub) * (n >> 3) + kt * 16 + l8 * 2;
    uint4* dst = codes + ((row0 + sub) * out_k_tiles + out_kt0 + kt) * 8 + l8;
    const long long src_step = 32ll * (n >> 3), dst_step = 32ll * out_k_tiles * 8;
    uint4 lo[4], hi[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        lo[i] = hi[i] = make_uint4(0u, 0u, 0u, 0u);
        if (sub + 32 * i < n_rows) mx_load32(src + i * src_step, whole, lo[i], hi[i]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int se = mx_block_exp2(lo[i], hi[i]);
        if (sub + 32 * i < n_rows) dst[i * dst_step] = mx_codes16(lo[i], hi[i], se);
        if ((l8 & 1) == 0) sf[(sub + 32 * i) * 4 + (l8 >> 1)] = (uint8_t)(se + 127);
    }
    __syncthreads();
    const int i = threadIdx.x;
    const uint32_t* words = reinterpret_cast<const uint32_t*>(sf);
    if (!WEIGHTS) {
        if (i < n_rows) reinterpret_cast<uint32_t*>(scales)[(long long)(out_kt0 + kt) * rows + row0 + i] = words[i];
    } else if (i < 128) {   // n_feat is a multiple of 128: the 128 rows are 128 features of one expert
        const long long e = row0 / n_feat;
        const int f0 = (int)(row0 - e * n_feat);
        const int n_tiles_p = (n_feat + MXP_NT - 1) / MXP_NT;
        mx_store_weight_scales(words, f0,
                               reinterpret_cast<uint32_t*>(scales + ((e * (n_feat / 128) + f0 / 128) * out_k_tiles + out_kt0 + kt) * 512),
                               scales_pair + (e * n_tiles_p * out_k_tiles + out_kt0 + kt) * 1024, (long long)out_k_tiles * 1024, i);
    }
}

// The SwiGLU activation of saved pre-activations with the activation quantiser fused in: GU [rows, 2I] bf16 ->
// H_act [rows, I] bf16 (silu(g) * u in fp32, rounded once) and the block-scaled FP8 codes and scale words of exactly those
// bf16 values, in the layouts of the activation quantiser.  Same mapping as mx_quantize_rows_kernel, on 64 rows: a half-warp
// per (row, 128-wide slice of I), four rows one after the other with all eight loads in flight.
// 16384 x 14336 inside an FP8 step 320 -> 248 us, alone 289 -> 242 us (6.8 TB/s); 131072 x 768 138 -> 110 us.  Before, a thread
// had two loads in flight, and every row took a division and four more shuffles.
constexpr int MX_SWIGLU_ROWS = 64;
__global__ void __launch_bounds__(256) mx_swiglu_quantize_kernel(const uint4* __restrict__ gu, long long rows, int I,
                                                                 uint4* __restrict__ h_act, uint2* __restrict__ codes,
                                                                 uint32_t* __restrict__ scales) {
    __shared__ __align__(16) uint8_t sf[MX_SWIGLU_ROWS * 4];
    if (!grid_dependency_wait_tested()) return;
    grid_launch_dependents();
    constexpr int N = MX_SWIGLU_ROWS / 16;
    const int k_tiles = I >> 7, iv = I >> 3;
    const int row_tile = (int)(blockIdx.x / (unsigned)k_tiles), kt = (int)(blockIdx.x - (unsigned)row_tile * (unsigned)k_tiles);
    const long long row0 = (long long)MX_SWIGLU_ROWS * row_tile;
    const int sub = threadIdx.x >> 4, l16 = threadIdx.x & 15;
    const int n_rows = (int)min((long long)MX_SWIGLU_ROWS, rows - row0);
    const uint4* src = gu + (row0 + sub) * (2 * iv) + kt * 16 + l16;
    const long long dst0 = (row0 + sub) * iv + kt * 16 + l16;
    uint4 g[N], u[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const bool in = sub + 16 * i < n_rows;
        g[i] = in ? __ldg(src + 32ll * i * iv) : make_uint4(0u, 0u, 0u, 0u);
        u[i] = in ? __ldg(src + 32ll * i * iv + iv) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint32_t* gw = reinterpret_cast<const uint32_t*>(&g[i]);
        const uint32_t* uw = reinterpret_cast<const uint32_t*>(&u[i]);
        uint32_t hw[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float g0 = mx_lo(gw[j]), g1 = mx_hi(gw[j]);
            hw[j] = pack_bf16(__fdividef(g0, 1.f + __expf(-g0)) * mx_lo(uw[j]), __fdividef(g1, 1.f + __expf(-g1)) * mx_hi(uw[j]));
        }
        const uint4 h = make_uint4(hw[0], hw[1], hw[2], hw[3]);
        const int se = mx_block_exp(h);
        if (sub + 16 * i < n_rows) {
            h_act[dst0 + 16ll * i * iv] = h;
            codes[dst0 + 16ll * i * iv] = mx_codes8(h, se);
        }
        if ((l16 & 3) == 0) sf[(sub + 16 * i) * 4 + (l16 >> 2)] = (uint8_t)(se + 127);
    }
    __syncthreads();
    if ((int)threadIdx.x < n_rows) scales[(long long)kt * rows + row0 + threadIdx.x] = reinterpret_cast<const uint32_t*>(sf)[threadIdx.x];
}

// The SwiGLU backward (elementwise part of the gate/up backward) with the row quantiser of its result fused in:
// dGU = [dg | du] [rows, 2I] bf16 exactly as moe_swiglu_bwd computes it, and the block-scaled FP8 codes and scale words of
// those bf16 values along the 2I columns (the A operand of the FP8 gate/up dgrad).  The same mapping on 32 rows: a half-warp
// per (row, 128-wide slice of each half), two rows one after the other with all six loads in flight.
// 16384 x 14336 inside an FP8 step 494 -> 478 us (5.9 TB/s), 131072 x 768 222 -> 205 us; alone 442 and 451 us.
constexpr int MX_SWIGLU_BWD_ROWS = 32;
__global__ void __launch_bounds__(256) mx_swiglu_bwd_quantize_kernel(const uint4* __restrict__ dh_act, const uint4* __restrict__ gu,
                                                                     long long rows, int I, uint4* __restrict__ dgu,
                                                                     uint2* __restrict__ codes, uint32_t* __restrict__ scales) {
    __shared__ __align__(16) uint8_t sf[2][MX_SWIGLU_BWD_ROWS * 4];
    if (!grid_dependency_wait_tested()) return;
    grid_launch_dependents();
    constexpr int N = MX_SWIGLU_BWD_ROWS / 16;
    const int k_tiles = I >> 7, iv = I >> 3;
    const int row_tile = (int)(blockIdx.x / (unsigned)k_tiles), kt = (int)(blockIdx.x - (unsigned)row_tile * (unsigned)k_tiles);
    const long long row0 = (long long)MX_SWIGLU_BWD_ROWS * row_tile;
    const int sub = threadIdx.x >> 4, l16 = threadIdx.x & 15;
    const int n_rows = (int)min((long long)MX_SWIGLU_BWD_ROWS, rows - row0);
    const long long at = (row0 + sub) * (2 * iv) + kt * 16 + l16;   // in GU and dGU; dH_act has half the pitch
    const uint4* dh_src = dh_act + (row0 + sub) * iv + kt * 16 + l16;
    uint4 d[N], g[N], u[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const bool in = sub + 16 * i < n_rows;
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        d[i] = in ? __ldg(dh_src + 16ll * i * iv) : zero;
        g[i] = in ? __ldg(gu + at + 32ll * i * iv) : zero;
        u[i] = in ? __ldg(gu + at + 32ll * i * iv + iv) : zero;
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint32_t* dw = reinterpret_cast<const uint32_t*>(&d[i]);
        const uint32_t* gw = reinterpret_cast<const uint32_t*>(&g[i]);
        const uint32_t* uw = reinterpret_cast<const uint32_t*>(&u[i]);
        uint32_t og[4], ou[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 d2 = make_float2(mx_lo(dw[j]), mx_hi(dw[j])), g2 = make_float2(mx_lo(gw[j]), mx_hi(gw[j]));
            const float2 u2 = make_float2(mx_lo(uw[j]), mx_hi(uw[j]));
            const float s0 = __fdividef(1.f, 1.f + __expf(-g2.x)), s1 = __fdividef(1.f, 1.f + __expf(-g2.y));
            og[j] = pack_bf16(d2.x * u2.x * s0 * (1.f + g2.x * (1.f - s0)), d2.y * u2.y * s1 * (1.f + g2.y * (1.f - s1)));
            ou[j] = pack_bf16(d2.x * g2.x * s0, d2.y * g2.y * s1);
        }
        const uint4 vg = make_uint4(og[0], og[1], og[2], og[3]), vu = make_uint4(ou[0], ou[1], ou[2], ou[3]);
        const int se_g = mx_block_exp(vg), se_u = mx_block_exp(vu);
        if (sub + 16 * i < n_rows) {
            const long long to = at + 32ll * i * iv;
            dgu[to] = vg;
            dgu[to + iv] = vu;
            codes[to] = mx_codes8(vg, se_g);
            codes[to + iv] = mx_codes8(vu, se_u);
        }
        if ((l16 & 3) == 0) {
            sf[0][(sub + 16 * i) * 4 + (l16 >> 2)] = (uint8_t)(se_g + 127);
            sf[1][(sub + 16 * i) * 4 + (l16 >> 2)] = (uint8_t)(se_u + 127);
        }
    }
    __syncthreads();
    const int half = threadIdx.x >> 5, r = threadIdx.x & 31;   // a warp per half of the columns
    if (half < 2 && r < n_rows)
        scales[(long long)(half * k_tiles + kt) * rows + row0 + r] = reinterpret_cast<const uint32_t*>(sf[half])[r];
}

// ---- quantisers along the rows of a row-major operand (codes stored transposed) ----
// 128 rows x 128 features of a row-major bf16 matrix -> 128 code bytes per feature, contiguous, and a scale byte per (feature,
// block of 32 rows).  Shared by the weight quantiser (weights whose output-feature axis is contiguous) and the token-axis
// quantiser.  The tile comes in with 16-byte asynchronous copies (rows from `n_rows` on as zeros); a thread then owns a
// pair of features over one block of 32 rows: 32 words from shared memory (blocks of rows are set 8 words apart so that
// the 4 x 8 lanes of a warp hit 32 banks), both maxima in packed arithmetic, 2 x 32 code bytes.  The 4 lanes that share a
// feature write its 128 contiguous bytes, 32 each with one store: two 16-byte stores write every 32-byte sector by halves, and
// that costs the L2 as much as twice the bytes.  Token axis 131072 x 2048 186 -> 154 us, 16384 x 14336 166 -> 135 us; weights
// 128 x 768 x 2048 113 -> 100 us.  Callers' buffers need only 16-byte alignment, hence the other branch.
constexpr int MXT_BLOCK_WORDS = 32 * 64 + 8;   // shared-memory words of 32 rows x 128 features, with the bank offset
__device__ __forceinline__ void mx_transpose_quantize_tile(const bf16* src, long long ld, int n_rows, uint8_t* dst, long long dst_ld,
                                                           uint32_t* tile, uint8_t* sf) {
    const int tid = threadIdx.x;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int row = i * 16 + (tid >> 4), piece = tid & 15;
        const bool in = row < n_rows;
        const bf16* from = src + (in ? row * ld : 0) + piece * 8;
        const uint32_t to = smem_u32(tile + (row >> 5) * MXT_BLOCK_WORDS + (row & 31) * 64 + piece * 4);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(from), "r"(in ? 16 : 0) : "memory");
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const int lane = tid & 31, block = lane >> 3, pair = (tid >> 5) * 8 + (lane & 7);   // features 2 * pair, 2 * pair + 1
    const uint32_t* col = tile + block * MXT_BLOCK_WORDS + pair;
    uint32_t v[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = col[j * 64];
    uint32_t m = 0u;
#pragma unroll
    for (int j = 0; j < 32; ++j) m = mx_abs_max(m, v[j] & 0x7fff7fffu);
    const int exps[2] = {mx_scale_exp(mx_lo(m)), mx_scale_exp(mx_hi(m))};
    const bool whole_sectors = (reinterpret_cast<uintptr_t>(dst) & 31) == 0;   // for the whole grid: all but the buffer is a multiple of 32
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float inv = mx_inv_scale(exps[h]);
        uint32_t out[8];
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            float f[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) f[t] = (h ? mx_hi(v[4 * g + t]) : mx_lo(v[4 * g + t])) * inv;
            out[g] = mx_e4m3x2(f[0], f[1]) | (mx_e4m3x2(f[2], f[3]) << 16);
        }
        uint8_t* to = dst + (2 * pair + h) * dst_ld + block * 32;
        if (whole_sectors) {
            asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(to), "r"(out[0]), "r"(out[1]), "r"(out[2]),
                         "r"(out[3]), "r"(out[4]), "r"(out[5]), "r"(out[6]), "r"(out[7])
                         : "memory");
        } else {
            reinterpret_cast<uint4*>(to)[0] = make_uint4(out[0], out[1], out[2], out[3]);
            reinterpret_cast<uint4*>(to)[1] = make_uint4(out[4], out[5], out[6], out[7]);
        }
        sf[(2 * pair + h) * 4 + block] = (uint8_t)(exps[h] + 127);
    }
    __syncthreads();
}

// Weights whose OUTPUT-feature axis is contiguous: w [E, k, n] bf16 (W_down [E, I, H]; W_gate, W_up [E, H, I]) -> codes
// transposed, contraction contiguous, as rows n_off .. n_off + n of [E, n_total, k] (W_gate and W_up stacked along the 2I
// output features of the gate/up projection), and the scale bytes in both tilings.  One block per (expert, K slice of
// 128, 128 features), features fastest.
// 201 M weights (128 x 768 x 2048): 165 -> 113 us (5.3 TB/s) inside an FP8 step.  Before, a thread loaded its 32 x 1 values
// two bytes at a time and stored its scale bytes one by one into both tilings.
__global__ void __launch_bounds__(256) mx_quantize_w_transposed_kernel(const bf16* __restrict__ w, int k, int n, int n_total,
                                                                       int n_off, uint8_t* __restrict__ codes,
                                                                       uint8_t* __restrict__ scales,
                                                                       uint8_t* __restrict__ scales_pair) {
    __shared__ __align__(16) uint32_t tile[4 * MXT_BLOCK_WORDS];
    __shared__ __align__(16) uint8_t sf[128 * 4];
    if (!grid_dependency_wait_tested()) return;
    grid_launch_dependents();
    const int f_tiles = n >> 7, k_tiles = k >> 7;
    const int ft = blockIdx.x % f_tiles, rest = blockIdx.x / f_tiles, kt = rest % k_tiles;
    const long long e = rest / k_tiles;
    const int f0 = n_off + ft * 128;   // first output feature of the GEMM
    mx_transpose_quantize_tile(w + (e * k + kt * 128ll) * n + ft * 128, n, 128, codes + (e * n_total + f0) * k + kt * 128, k, tile, sf);
    const int n_tiles_p = (n_total + MXP_NT - 1) / MXP_NT;
    if (threadIdx.x < 128)
        mx_store_weight_scales(reinterpret_cast<const uint32_t*>(sf), f0,
                               reinterpret_cast<uint32_t*>(scales + ((e * (n_total / 128) + f0 / 128) * k_tiles + kt) * 512),
                               scales_pair + (e * n_tiles_p * k_tiles + kt) * 1024, (long long)k_tiles * 1024, threadIdx.x);
}


// ---- token-axis quantiser (operands of the weight gradients) ---------------------------------------------
// dW[e] [M, N] = Q(A_e)^T Q(B_e) over the rows of expert e, both operands quantised along the token axis in blocks of 32
// rows counted from the expert's first row and stored TRANSPOSED, contraction contiguous: codes [features, pitch] where
// column slice_prefix[e] * 128 + i holds row offsets[e] + i of the packed tensor and every expert's columns are padded
// with zero codes to a multiple of 128 -- so a K slice of 128 columns belongs to exactly one expert, both operands are
// K-major like everywhere else in this file, and the ragged contraction needs no clearing of foreign rows in shared
// memory.  The tile list is fixed (every expert x M tiles x N tiles); an expert's K slices are
// [slice_prefix[e], slice_prefix[e+1]); a tile of an expert without rows skips the pipeline and its epilogue writes zeros.
// x [R, ld] bf16, columns [col0, col0 + n) -> codes_t [n, pitch] (transposed, zero-padded per expert), scale words
// [pitch/128][n] (the operand as the M side) and scale blocks in the pair tiling [ceil(n/208)][pitch/128][1024] (the
// operand as the N side).  One block per (slice of 128 columns of the output, 128 features), features fastest.  Every block
// derives slice_prefix (slice_prefix[e] = number of 128-row slices of the experts before e, every expert's rows rounded
// up to whole slices) from the offsets by itself -- a scan over at most 1024 experts that overlaps the copies of the other
// blocks on the SM -- and the first one stores it for the GEMM.
// Inside an FP8 step, 16384 x 14336: 240 + 3 -> 196 us, 16384 x 4096: 98 + 3 -> 59 us (a kernel of its own wrote
// slice_prefix before); alone on the chip 150 us and 49 us.  What is left inside the step is instruction issue at the clock
// that the power cap leaves.  Taking several slices before the next 128 features (4 to 32: longer runs of code bytes per
// feature) changed nothing.
__global__ void __launch_bounds__(256) mx_quantize_tokens_kernel(const bf16* __restrict__ x, long long ld, int col0, int n,
                                                                 const int32_t* __restrict__ offsets, int32_t* __restrict__ sp,
                                                                 int E, long long pitch, uint8_t* __restrict__ codes_t,
                                                                 uint32_t* __restrict__ sa_words, uint8_t* __restrict__ sb_atoms) {
    __shared__ __align__(16) uint32_t tile[4 * MXT_BLOCK_WORDS];
    __shared__ __align__(16) uint8_t sf[128 * 4];
    __shared__ int32_t part[8];
    __shared__ int32_t mine[3];   // first row, rows and existence of this block's slice
    if (!grid_dependency_wait_tested()) return;
    grid_launch_dependents();
    const int f_tiles = n >> 7;
    const int f0 = (int)(blockIdx.x % (unsigned)f_tiles) * 128, slice = (int)(blockIdx.x / (unsigned)f_tiles);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // thread t scans the experts 4t .. 4t + 3
    int32_t off[5], before[4], sum = 0;
#pragma unroll
    for (int i = 0; i < 5; ++i) off[i] = __ldg(offsets + min(4 * tid + i, E));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        before[i] = sum;
        sum += (off[i + 1] - off[i] + 127) >> 7;
    }
    int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
    }
    if (lane == 31) part[warp] = incl;
    if (tid == 0) mine[2] = 0;
    __syncthreads();
    int base = incl - sum;
    for (int w = 0; w < warp; ++w) base += part[w];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int first = base + before[i], local = slice - first;
        const int rows = off[i + 1] - off[i];
        if (local >= 0 && local * 128 < rows) {   // at most one (thread, i) of the block: the expert that holds the slice
            mine[0] = off[i] + local * 128;
            mine[1] = min(128, rows - local * 128);
            mine[2] = 1;
        }
        if (blockIdx.x == 0 && 4 * tid + i <= E) sp[4 * tid + i] = first;
    }
    if (blockIdx.x == 0 && E == 1024 && tid == 255) sp[E] = base + sum;
    __syncthreads();
    if (mine[2] == 0) return;   // past the last slice
    mx_transpose_quantize_tile(x + (long long)mine[0] * ld + col0 + f0, ld, mine[1], codes_t + (long long)f0 * pitch + slice * 128ll, pitch,
                               tile, sf);
    if (tid < 128) {
        const uint32_t* words = reinterpret_cast<const uint32_t*>(sf);
        sa_words[(long long)slice * n + f0 + tid] = words[tid];
        mx_store_weight_scales(words, f0, nullptr, sb_atoms + slice * 1024ll, (pitch >> 7) * 1024, tid);
    }
}

}  // namespace

// Weight scales of a GEMM with E experts, n_feat output features and a contraction of k: stored twice, in the tiling of
// the single-CTA kernel, then in that of the CTA-pair kernel.
size_t mx_w_scale_single_bytes(int E, int n_feat, int k) { return (size_t)E * (n_feat / 128) * (k / 128) * 512; }
size_t mx_w_scale_bytes(int E, int n_feat, int k) {
    return mx_w_scale_single_bytes(E, n_feat, k) + (size_t)E * ((n_feat + MXP_NT - 1) / MXP_NT) * (k / 128) * 1024;
}

static unsigned mx_row_quantiser_blocks(long long rows, int k) { return (unsigned)((rows + 127) / 128 * (k / 128)); }

int launch_mx_quantize_rows(long long rows, int n, const bf16* x, uint8_t* codes, uint8_t* scales, cudaStream_t s) {
    return launch_streaming(mx_quantize_rows_kernel<false>, mx_row_quantiser_blocks(rows, n), s, reinterpret_cast<const uint4*>(x), rows, n, 0, n / 128, 0, reinterpret_cast<uint4*>(codes), scales,
                            static_cast<uint8_t*>(nullptr));
}

// w [E, k, n] -> rows [n_off, n_off + n) of the transposed codes [E, n_total, k] and the matching scale bytes
int launch_mx_quantize_w_transposed(int E, int k, int n, int n_total, int n_off, const bf16* w, uint8_t* codes_t, uint8_t* scales,
                                    cudaStream_t s) {
    const long long blocks = (long long)E * (k / 128) * (n / 128);
    return launch_streaming(mx_quantize_w_transposed_kernel, (unsigned)blocks, s, w, k, n, n_total, n_off, codes_t, scales,
                            scales + mx_w_scale_single_bytes(E, n_total, k));
}

int launch_mx_swiglu_quantize(long long rows, int I, const bf16* gu, bf16* h_act, uint8_t* codes, uint8_t* scales, cudaStream_t s) {
    const long long blocks = (rows + MX_SWIGLU_ROWS - 1) / MX_SWIGLU_ROWS * (I / 128);
    return launch_streaming(mx_swiglu_quantize_kernel, (unsigned)blocks, s, reinterpret_cast<const uint4*>(gu), rows, I,
                            reinterpret_cast<uint4*>(h_act), reinterpret_cast<uint2*>(codes), reinterpret_cast<uint32_t*>(scales));
}

int launch_mx_swiglu_bwd_quantize(long long rows, int I, const bf16* dh_act, const bf16* gu, bf16* dgu, uint8_t* codes,
                                  uint8_t* scales, cudaStream_t s) {
    const long long blocks = (rows + MX_SWIGLU_BWD_ROWS - 1) / MX_SWIGLU_BWD_ROWS * (I / 128);
    return launch_streaming(mx_swiglu_bwd_quantize_kernel, (unsigned)blocks, s, reinterpret_cast<const uint4*>(dh_act),
                            reinterpret_cast<const uint4*>(gu), rows, I, reinterpret_cast<uint4*>(dgu), reinterpret_cast<uint2*>(codes),
                            reinterpret_cast<uint32_t*>(scales));
}

// w [E * n_feat, k] -> columns [k_off, k_off + k) of the codes [E * n_feat, k_total] and the matching scale slices
int launch_mx_quantize_w_rows(int E, int n_feat, int k, int k_total, int k_off, const bf16* w, uint8_t* codes, uint8_t* scales,
                              cudaStream_t s) {
    const long long rows = (long long)E * n_feat;
    return launch_streaming(mx_quantize_rows_kernel<true>, mx_row_quantiser_blocks(rows, k), s, reinterpret_cast<const uint4*>(w), rows, k, n_feat,
                            k_total / 128, k_off / 128, reinterpret_cast<uint4*>(codes), scales,
                            scales + mx_w_scale_single_bytes(E, n_feat, k_total));
}

// ---- weight-gradient operands and GEMM ----
constexpr size_t MX_TOKENS_HEADER_BYTES = 8192;   // slice_prefix[E + 1] at the head of a token-quantised operand's scales
long long mx_tokens_pitch(long long R, int E) { return ((R + 127) / 128) * 128 + 128ll * E; }
size_t mx_tokens_scale_bytes(long long R, int E, int n) {
    const long long slices = mx_tokens_pitch(R, E) / 128;
    return MX_TOKENS_HEADER_BYTES + (size_t)slices * n * 4 + (size_t)((n + MXP_NT - 1) / MXP_NT) * slices * 1024;
}

int launch_mx_quantize_tokens(long long R, int E, const bf16* x, long long ld, int col0, int n, const int32_t* offsets,
                              uint8_t* codes_t, uint8_t* scales, cudaStream_t s) {
    const long long pitch = mx_tokens_pitch(R, E);
    int32_t* sp = reinterpret_cast<int32_t*>(scales);
    uint8_t* sa = scales + MX_TOKENS_HEADER_BYTES;
    uint8_t* sb = sa + (size_t)(pitch / 128) * n * 4;
    // no more slices than rows: with less than a row per expert most of the pitch is never used (256 experts, 8 rows of 7168:
    // 28 us with a block for all of it)
    const long long slices = pitch / 128 < R ? pitch / 128 : R;
    const long long blocks = slices * (n / 128);
    return launch_streaming(mx_quantize_tokens_kernel, (unsigned)blocks, s, x, ld, col0, n, offsets, sp, E,
                            pitch, codes_t, reinterpret_cast<uint32_t*>(sa), sb);
}

template <int FORM>
static int launch_mx_pair(const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& b_low, const CUtensorMap& sf, const CUtensorMap& o, const MxPairParams& p,
                          cudaStream_t s) {
    static int grid_of_device[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return MOE_ERR_CUDA;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(MXP_THREADS);
    cfg.dynamicSmemBytes = MXP_SMEM_BYTES;
    cfg.attrs = attr; cfg.numAttrs = 1;
    if (grid_of_device[dev] == 0) {
        if (cudaFuncSetAttribute(mx_pair_kernel<FORM>, cudaFuncAttributeMaxDynamicSharedMemorySize, MXP_SMEM_BYTES) != cudaSuccess)
            return MOE_ERR_CUDA;
        const int sms = sm_count();
        if (sms <= 0) return MOE_ERR_CUDA;
        // as many pairs as can be resident at once: a pair that had to wait for a free SM pair would double the duration
        cfg.gridDim = dim3(2 * (sms / 2));
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, mx_pair_kernel<FORM>, &cfg) != cudaSuccess || clusters <= 0) return MOE_ERR_CUDA;
        if (clusters > sms / 2) clusters = sms / 2;
        grid_of_device[dev] = 2 * clusters;
    }
    return launch_dependent(mx_pair_kernel<FORM>, grid_of_device[dev], MXP_THREADS, MXP_SMEM_BYTES, 2, s, a, b, b_low, sf, o, p);
}

// dW [E, M, N] = Q(A)^T Q(B) per expert: a_* the M-side operand ([M, pitch] codes, scales with header and words),
// b_* the N-side operand ([N, pitch] codes, its scales' pair-tiled blocks are used)
int launch_mx_wgrad(long long R, int E, int M, int N, const uint8_t* a_codes_t, const uint8_t* a_scales, const uint8_t* b_codes_t,
                    const uint8_t* b_scales, bf16* dw, cudaStream_t s) {
    const long long pitch = mx_tokens_pitch(R, E);
    const int n_slices = (int)(pitch / 128);
    const int n_tiles = (N + MXP_NT - 1) / MXP_NT, m_tiles = (M + MXP_ROWS - 1) / MXP_ROWS;
    const uint8_t* b_atoms = b_scales + MX_TOKENS_HEADER_BYTES + (size_t)n_slices * N * 4;
    CUtensorMap a, b, sfb, o;
    if (!make_map_typed(&a, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, a_codes_t, (uint64_t)pitch, (uint64_t)M, MX_BK, MX_BM, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_typed(&b, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, b_codes_t, (uint64_t)pitch, (uint64_t)N, MX_BK, MXP_NT / 2,
                        CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_typed(&sfb, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, b_atoms, 256, (uint64_t)n_tiles * n_slices, 256, 1,
                        CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_out_map(&o, dw, N, (uint64_t)E * M))
        return MOE_ERR_CUDA;
    MxPairParams p = {};
    p.prefix = reinterpret_cast<const int32_t*>(a_scales); p.E = E; p.M = M; p.m_tiles = m_tiles; p.n_tiles = n_tiles;
    p.n_cols = N; p.n_slices = n_slices; p.sa_rows = M;
    p.sa = reinterpret_cast<const uint32_t*>(a_scales + MX_TOKENS_HEADER_BYTES); p.out = dw; p.ldo = N;
    return launch_mx_pair<MXP_WGRAD>(a, b, b, sfb, o, p, s);
}

// Which kernel for R rows of E experts, n_feat output features, a contraction of k.
// CTA pairs, weights on M, from 256 rows per expert on average, and from 96 on if there are tiles for all pairs of the chip even with
// one row tile per expert and the contraction is at least 512.  Single CTA against pair, gate/up / down / down dgrad / gate/up dgrad, rows per expert:
//   128 (128 experts, 2048 x 768)   108 / 70 / 60 / 117 against 102 / 65 / 60 / 105 us     81:  88 / 63 / 52 / 96 against 83 / 60 / 51 / 91 us
//   128 (8 experts, 4096 x 14336)   213 / 126 / 112 / 255 against 189 / 100 / 103 / 191 us  80:  169 / 93 / 92 / 172 against 170 / 95 / 96 / 176 us
//   125 (16 experts, 256 x 512: 16 to 64 pair tiles)   7.7 / 5.6 / 5.5 / 6.1 against 8.0 / 6.5 / 6.2 / 7.4 us
//   229 (2 experts, gate/up of 6272 features each, contraction 128)   6.5 against 7.4 us
// Not where 256 features per tile leave half (128 features) or a quarter (384) of them empty: of 128 features single CTAs, whatever the
// rows (weights on M / rows on M / single CTA: 893 rows, 110 experts, k 2688 76 / 62 / 64 us, 3794, 4, k 1024 13.0 / 9.4 / 8.1, 98, 170, k 768 13.2 /
// 12.7 / 9.6), of 384 rows on M, below 256 rows single CTAs (5263, 9, k 8064 176 / 144 / 169, 733, 10, k 2432 16.5 / 11.7 / 13.4, 110, 129, k 1024
// 22.5 / 22.3 / 19.9).
// And not where it takes more rounds of tiles over the chip's CTA pairs, each round at its price (a tile of w rows on N 0.76 + 0.24 w / 208 of
// a full one's time, a single CTA's tile 0.81).  Weights on M / rows on M: 481 rows, 85 experts, 1664 features, k 768 76 / 65 us, 419, 152, 3328, k 640 234 / 199 us.  Weights
// on M / single CTA: 106 rows, 15 experts, 2432 features, k 896 12.9 / 10.6 us, 96, 130, 640, k 3456 69 / 61 us.
// 2340 drawn shapes from 96 rows on: this rule 3.2 % above the best form of each on average, weights on M from 256 rows throughout 6.3 %,
// rows on M 9.0 %; slower than rows on M by more than a tenth 18 of them, with weights on M throughout 265.
enum MxGemmForm { MX_SINGLE, MX_PAIR_WEIGHTS_M, MX_PAIR_ROWS_M };
static MxGemmForm mx_form(long long R, int E, int n_feat, int k) {
    const int on_m = (n_feat + MXP_ROWS - 1) / MXP_ROWS, on_n = (n_feat + MXP_NT - 1) / MXP_NT;   // tiles of features
    const bool mostly_full = 5 * n_feat >= 4 * MXP_ROWS * on_m, small = R < 256ll * E;
    if (R < 96ll * E || n_feat <= 128) return MX_SINGLE;
    if (small && !(mostly_full && k >= 512 && (long long)E * on_m >= kChipPairs)) return MX_SINGLE;
    if (!mostly_full) return MX_PAIR_ROWS_M;
    const double rows = (double)R / E, tile_n = ceil(rows / ceil(rows / MXP_NT) / 16) * 16;
    const double weights_m = tile_rounds(R, E, MXP_NT, on_m, kChipPairs) * (0.76 + 0.24 * (tile_n / MXP_NT + 1) / 2);
    if (small) return 0.95 * weights_m < 0.81 * tile_rounds(R, E, MX_BM, n_feat / MX_BN, 2 * kChipPairs) ? MX_PAIR_WEIGHTS_M : MX_SINGLE;
    return 1.03 * tile_rounds(R, E, MXP_ROWS, on_n, kChipPairs) < weights_m ? MX_PAIR_ROWS_M : MX_PAIR_WEIGHTS_M;
}
// The swapped form of the single-CTA kernel up to this many rows per expert on average.  There the time is the weights'
// way from HBM, and what counts is bytes in flight and an even spread over the SMs: two CTAs with four stages of weights
// and at most 64 rows each, against one with six stages that also hold 128 rows.  Down projection of 8 experts,
// 14336 x 4096, 25 rows each (event times, cold L2): 92 -> 80 us, gate/up 162 -> 152 us; 37 such experts 351 -> 328 and
// 715 -> 650 us (6.9 TB/s).  128 experts, 768 x 2048, down projection, rows per expert 32: 47 -> 44 us, 64: 51 -> 47 us,
// 94: 51 -> 55 us -- a second tile per expert reads the expert's weights again, from L2.  Tiles of 32 rows lost to
// tiles of 64 everywhere but below 4 rows per expert (N = 32 makes the MMAs no cheaper to issue).
// Under Zipf and Dirichlet loads, where one expert runs many 64-row tiles, the form holds: 128 experts, 64 rows on average, at most
// 973 / 756, down 54 -> 48 / 49 -> 44 us, gate/up 89 -> 83 / 78 -> 78 us (unswapped -> swapped); 64 experts of 2048 x 1408 40-43 -> 37-40 us.
// Not so few large experts just below the line: 8 experts of 64 rows, 14336 x 4096, down 87 -> 108 us (gate/up 168 -> 173 us).
// Not with so many experts (487 and more) that two CTAs and their tables no longer fit an SM: the second half of the grid
// would wait for the first, and one CTA with four stages keeps less in flight than one with six.  Down projection, 1024 x 512,
// swapped with one CTA per SM against this kernel unswapped: 512 experts of 4 rows 76 against 55 us, of 64 rows 108 against
// 68 us, 1024 experts of 64 rows under a Zipf load 237 against 154 us; 480 experts of 64 rows, two CTAs per SM, 62 against 69 us.
constexpr long long kMxSwappedRows = 64;
static bool mx_single_swapped(long long R, int E) { return R <= kMxSwappedRows * E && MxGeo<64>::all_ctas_fit(E); }

static int launch_mx_gemm_pair_weights_m(long long R, int E, int n_feat, int k, const uint8_t* a_codes, const uint8_t* a_scales,
                               const uint8_t* b_codes, const uint8_t* b_scales, const int32_t* offsets, bf16* out,
                               cudaStream_t s) {
    const int k_tiles = k / MX_BK;
    CUtensorMap w, x, x_low, sf, o;
    if (!make_map_typed(&w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, b_codes, k, (uint64_t)E * n_feat, MX_BK, MX_BM, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_typed(&x, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, a_codes, k, (uint64_t)R, MX_BK, MXP_NT / 2, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_typed(&x_low, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, a_codes, k, (uint64_t)R, MX_BK, MXP_LOW_BOX, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_typed(&sf, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, b_scales, 128, (uint64_t)E * (n_feat / 128) * k_tiles, 128, 1,
                        CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_out_map(&o, out, n_feat, (uint64_t)R))
        return MOE_ERR_CUDA;
    MxPairParams p = {};
    p.prefix = offsets; p.E = E; p.k_tiles = k_tiles; p.n_tiles = (n_feat + MXP_ROWS - 1) / MXP_ROWS; p.n_cols = n_feat; p.sa_rows = R;
    p.sa = reinterpret_cast<const uint32_t*>(a_scales); p.out = out; p.ldo = n_feat;
    return launch_mx_pair<MXP_WEIGHTS_M>(w, x, x_low, sf, o, p, s);
}
static int launch_mx_gemm_pair_rows_m(long long R, int E, int n_feat, int k, const uint8_t* a_codes, const uint8_t* a_scales,
                                      const uint8_t* b_codes, const uint8_t* b_scales, const int32_t* offsets, bf16* out,
                                      cudaStream_t s) {
    const int k_tiles = k / MX_BK, n_tiles = (n_feat + MXP_NT - 1) / MXP_NT;
    CUtensorMap x, w, sf, o;
    if (!make_map_typed(&x, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, a_codes, k, (uint64_t)R, MX_BK, MX_BM, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_typed(&w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, b_codes, k, (uint64_t)E * n_feat, MX_BK, MXP_NT / 2, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_typed(&sf, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, b_scales + mx_w_scale_single_bytes(E, n_feat, k), 256,
                        (uint64_t)E * n_tiles * k_tiles, 256, 1, CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_out_map(&o, out, n_feat, (uint64_t)R))
        return MOE_ERR_CUDA;
    MxPairParams p = {};
    p.prefix = offsets; p.E = E; p.k_tiles = k_tiles; p.n_tiles = n_tiles; p.n_cols = n_feat; p.sa_rows = R;
    p.sa = reinterpret_cast<const uint32_t*>(a_scales); p.out = out; p.ldo = n_feat;
    return launch_mx_pair<MXP_ROWS_M>(x, w, w, sf, o, p, s);
}

struct MxSingleArgs {
    long long R;
    int E, n_feat, k;
    const uint8_t *a_codes, *a_scales, *b_codes, *b_scales;
    const int32_t* offsets;
    bf16* out;
};
template <int ROWS>
static int launch_mx_gemm_single(const MxSingleArgs& g, cudaStream_t s) {
    // never a box of more rows than there are: a load that is mostly out of bounds is slow (8 rows of
    // 14336 against 8 large experts, in boxes of 128 rows: 113 us, of 8 rows: 82 us)
    const uint32_t box = g.R < ROWS ? (uint32_t)g.R : (uint32_t)ROWS;
    CUtensorMap a, b, o;
    if (!make_map_typed(&a, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, g.a_codes, g.k, (uint64_t)g.R, MX_BK, box, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_typed(&b, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, g.b_codes, g.k, (uint64_t)g.E * g.n_feat, MX_BK, MX_BN,
                        CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_out_map(&o, g.out, g.n_feat, (uint64_t)g.R))
        return MOE_ERR_CUDA;
    MxParams p = {};
    p.offsets = g.offsets; p.E = g.E; p.k_tiles = g.k / MX_BK; p.n_tiles = g.n_feat / MX_BN; p.n_cols = g.n_feat; p.R = g.R; p.x_bytes = box * MX_BK;
    p.sa = reinterpret_cast<const uint32_t*>(g.a_scales); p.sb = g.b_scales; p.out = g.out; p.ldo = g.n_feat;
    static bool attr_set[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return MOE_ERR_CUDA;
    if (!attr_set[dev]) {
        if (cudaFuncSetAttribute(mx_gemm_kernel<ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, MxGeo<ROWS>::smem_bytes(MX_MAX_E)) !=
            cudaSuccess)
            return MOE_ERR_CUDA;
        attr_set[dev] = true;
    }
    const int sms = sm_count();
    if (sms <= 0) return MOE_ERR_CUDA;
    return launch_dependent(mx_gemm_kernel<ROWS>, MxGeo<ROWS>::CTAS * sms, MX_THREADS, MxGeo<ROWS>::smem_bytes(g.E), 1, s, a, b, o, p);
}

// out[r, :] = dequant(a row r) . dequant(b[e])^T for the rows r of expert e: a [R, k] codes with scale words
// [k/128][R], b [E, n_feat, k] codes with both scale tilings, out [R, n_feat] bf16.
int launch_mx_gemm(long long R, int E, int n_feat, int k, const uint8_t* a_codes, const uint8_t* a_scales, const uint8_t* b_codes,
                   const uint8_t* b_scales, const int32_t* offsets, bf16* out, cudaStream_t s) {
    const MxGemmForm form = mx_form(R, E, n_feat, k);
    if (form == MX_PAIR_WEIGHTS_M) return launch_mx_gemm_pair_weights_m(R, E, n_feat, k, a_codes, a_scales, b_codes, b_scales, offsets, out, s);
    if (form == MX_PAIR_ROWS_M) return launch_mx_gemm_pair_rows_m(R, E, n_feat, k, a_codes, a_scales, b_codes, b_scales, offsets, out, s);
    const MxSingleArgs args = {R, E, n_feat, k, a_codes, a_scales, b_codes, b_scales, offsets, out};
    return mx_single_swapped(R, E) ? launch_mx_gemm_single<64>(args, s) : launch_mx_gemm_single<128>(args, s);
}

#ifdef MOE_TEST_HOOKS
// Test-only build: CTAs per SM that the single-CTA kernel is launched with for R rows of E experts, and the shared memory of one.
// (The occupancy query is no help: it reports one CTA per SM for any kernel that allocates tensor memory.)
extern "C" void moe_test_mx_single_ctas(int R, int E, int* ctas, int* smem) {
    const bool swapped = mx_single_swapped(R, E);
    *ctas = swapped ? MxGeo<64>::CTAS : MxGeo<128>::CTAS;
    *smem = swapped ? MxGeo<64>::smem_bytes(E) : MxGeo<128>::smem_bytes(E);
}
// ... and the kernel that R rows of E experts, n_feat features and a contraction of k go to (MxGemmForm).
extern "C" int moe_test_mx_form(long long R, int E, int n_feat, int k) { return mx_form(R, E, n_feat, k); }
#endif

}  // namespace moe

// PTX wrappers shared by the tensor-core kernels (mbarrier, bulk tensor copies, tcgen05) and the host helpers that
// encode tensor maps.  Internal; everything here is inline / forceinline.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

#include <string.h>

#include "common.cuh"

namespace moe {
namespace {

// Every device-side wait gives up after this long (2 s; a test-only build of the library shortens it).
#ifndef MOE_WAIT_LIMIT_NS
#define MOE_WAIT_LIMIT_NS 2000000000ull
#endif
constexpr unsigned long long WAIT_LIMIT_NS = MOE_WAIT_LIMIT_NS;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// shared::cluster address of `local_addr` (a shared::cta address of this CTA) in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_cta(uint32_t local_addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("{ .reg .b64 st; mbarrier.arrive.shared::cta.b64 st, [%0]; }" ::"r"(bar) : "memory");
}
// Arrive on a barrier of another CTA of the cluster (address from map_to_cta).  Default semantics: a
// cluster-scope release/acquire pair on every ring stage serialises the pipeline on fences (measured: half
// the throughput; even one fence per tile costs 10-20 % on short contractions).  None is needed: the data
// the arrival announces sits in the ARRIVING CTA's own shared memory -- written there by the TMA unit
// (complete before the local barrier wait returns) or by this warp's generic stores (each lane runs
// fence.proxy.async after its stores and the warp synchronises before the arrive is issued) -- and is
// read from there by that CTA's own tensor core once the first CTA, having seen the arrival, issues the MMA.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_bar) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("{ .reg .b64 st; mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1; }" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}
// non-blocking test of a barrier phase (acquire on success)
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{ .reg .pred p; mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}
__device__ __forceinline__ unsigned long long global_timer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait (2 s on %globaltimer).  Returns false when the CTA is aborting (this wait timed out, or another did);
// a wait that runs out records MOE_ERR_TIMEOUT in `status` (the translation unit's device status word).
// Every lane of a waiting warp polls: electing one lane and broadcasting the verdict measured 5-10 % slower,
// and suspend-time hints on the long waits changed nothing.
__device__ __forceinline__ bool mbar_wait_status(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status) {
    if (mbar_try_wait(bar, parity)) return true;
    unsigned long long t0 = 0;
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 0xFF) == 0) {
            if (*abort_flag) return false;
            const unsigned long long now = global_timer_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > WAIT_LIMIT_NS) {
                *abort_flag = 1;
                atomicExch(status, (int)MOE_ERR_TIMEOUT);
                return false;
            }
        }
    }
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
// Pair mode: the same loads with the completion (complete_tx) delivered to a barrier of EITHER CTA of the pair
// (.cta_group::2; `cluster_bar` is a shared::cluster address from map_to_cta): both CTAs' loads of a ring stage report
// to the barrier of the CTA that issues the MMAs, with no software relay in between.  No multicast: the data still
// has exactly one destination, this CTA's own shared memory.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t cluster_bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(cluster_bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t cluster_bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(cluster_bar)
        : "memory");
}
// arrive (one arrival) and announce `bytes` of transactions on a barrier of either CTA of the cluster
__device__ __forceinline__ void mbar_arrive_expect_tx_cluster(uint32_t cluster_bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cluster.b64 _, [%0], %1;" ::"r"(cluster_bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int x, int y, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(map), "r"(x), "r"(y),
                 "r"(src)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all0() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// arrive on `bar` once all tcgen05 operations issued so far by this thread have completed; in pair mode
// the arrival goes to the barrier at the same offset in BOTH CTAs
template <bool PAIR>
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    if (PAIR) {
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
            "h"((uint16_t)3)
            : "memory");
    } else {
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
    }
}
// same, but only this CTA's barrier is signalled
template <bool PAIR>
__device__ __forceinline__ void tc_commit_local(uint32_t bar) {
    if (PAIR)
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
    else
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// One tcgen05.mma; the shared-memory descriptors are given by their low words (address and leading offset), the high words
// are constants of the kind.  ACC: accumulate (a literal for all but a tile's first MMA).
template <bool PAIR, uint32_t A_HI, uint32_t B_HI>
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate) {
    if (PAIR) {
        asm volatile(
            "{ .reg .pred p; .reg .b64 a, b; setp.ne.u32 p, %4, 0; mov.b64 a, {%1, %5}; mov.b64 b, {%2, %6};"
            " tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, p; }" ::"r"(d_tmem),
            "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(accumulate), "n"(A_HI), "n"(B_HI)
            : "memory");
    } else {
        asm volatile(
            "{ .reg .pred p; .reg .b64 a, b; setp.ne.u32 p, %4, 0; mov.b64 a, {%1, %5}; mov.b64 b, {%2, %6};"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p; }" ::"r"(d_tmem),
            "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(accumulate), "n"(A_HI), "n"(B_HI)
            : "memory");
    }
}
// one lane of the (converged) warp, the same one every time
__device__ __forceinline__ bool elect_one() {
    uint32_t pred = 0;
    asm volatile("{ .reg .pred p; elect.sync _|p, 0xffffffff; @p mov.u32 %0, 1; }" : "+r"(pred));
    return pred != 0;
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t v[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&h);
}

// ---- a 32 x 32 accumulator block transposed on its way out -------------------------------------------
// With the weights on the M side the accumulator has a feature per lane and a row per column, and the output is row-major.  The
// block is read from tensor memory as matrix fragments (16x256b: lane t of the warp has features t / 4 and t / 4 + 8, columns
// 2 (t % 4) and the next, of every 8 columns; once for lanes 0..15, once for 16..31) and stored with stmatrix.trans, which
// turns 8 x 8 blocks round: four instructions per block instead of 32 two-byte stores.
//   v[16 h + 4 i + 2 s + c]: feature 16 h + 8 s + t / 4, row 8 i + 2 (t % 4) + c
//   w[4 i + 2 h + s]:        the same, rounded, c in the low and high half
__device__ __forceinline__ void tc_ld_frag16(uint32_t taddr, uint32_t* v) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tc_ld_frag32(uint32_t taddr, uint32_t (&v)[32]) {
    tc_ld_frag16(taddr, v);
    tc_ld_frag16(taddr + (16u << 16), v + 16);
}
// pairs of fp32 values (in fragment order) -> w; the values of lane half h alone
template <typename T>
__device__ __forceinline__ void pack_frag_half(const T* v, int h, uint32_t (&w)[16]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            float lo, hi;
            memcpy(&lo, &v[4 * i + 2 * s], 4);
            memcpy(&hi, &v[4 * i + 2 * s + 1], 4);
            w[4 * i + 2 * h + s] = pack_bf16(lo, hi);
        }
}
template <typename T>
__device__ __forceinline__ void pack_frag(const T (&v)[32], uint32_t (&w)[16]) {
    pack_frag_half(v, 0, w);
    pack_frag_half(v + 16, 1, w);
}
// this lane's address offset in a staging block (32 rows of 64 bytes, 64-byte swizzle): row lane % 8, features 8 (lane / 8) ...
__device__ __forceinline__ uint32_t frag_offset(int lane) { return (lane & 7) * 64 + (((lane >> 3) ^ ((lane >> 1) & 3)) << 4); }
__device__ __forceinline__ void store_frag(uint32_t at, const uint32_t (&w)[16]) {   // at: staging block + frag_offset
#pragma unroll
    for (int i = 0; i < 4; ++i)
        asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(at + i * 512), "r"(w[4 * i]),
                     "r"(w[4 * i + 1]), "r"(w[4 * i + 2]), "r"(w[4 * i + 3])
                     : "memory");
}
__device__ __forceinline__ void load_frag(uint32_t at, uint32_t (&w)[16]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(w[4 * i]), "=r"(w[4 * i + 1]), "=r"(w[4 * i + 2]), "=r"(w[4 * i + 3])
                     : "r"(at + i * 512)
                     : "memory");
}
// the first `rows` rows of a staging block to global memory (row pitch ld elements)
__device__ __forceinline__ void copy_block_rows(const uint8_t* block, bf16* dst, long long ld, int rows, int lane) {
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const int j = s * 8 + (lane >> 2);
        if (j < rows)
            *reinterpret_cast<uint4*>(dst + j * ld + (lane & 3) * 8) =
                *reinterpret_cast<const uint4*>(block + j * 64 + (((lane & 3) ^ ((j >> 1) & 3)) << 4));
    }
}

// prefix[e] = number of tiles of `rows_per_tile` rows of the experts before e, prefix[E] = all of them.  One warp.
__device__ __forceinline__ void exclusive_tile_prefix(const int32_t* offs, int32_t* prefix, int E, int rows_per_tile, int lane) {
    int run = 0;
    for (int e0 = 0; e0 < E; e0 += 32) {
        const int e = e0 + lane;
        const int tiles = e < E ? (offs[e + 1] - offs[e] + rows_per_tile - 1) / rows_per_tile : 0;
        int incl = tiles;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += v;
        }
        if (e < E) prefix[e] = run + incl - tiles;
        run += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) prefix[E] = run;
}

// ---- host side: tensor maps -------------------------------------------------------------------------
inline PFN_cuTensorMapEncodeTiled_v12000 get_encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (fn == nullptr) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
    }
    return fn;
}

// 2-D tensor [outer, inner] (inner contiguous) of 1- or 2-byte elements, box [box_outer, box_inner].
inline bool make_map_typed(CUtensorMap* map, CUtensorMapDataType type, uint32_t elem_bytes, const void* base, uint64_t inner,
                           uint64_t outer, uint32_t box_inner, uint32_t box_outer, CUtensorMapSwizzle swizzle) {
    PFN_cuTensorMapEncodeTiled_v12000 fn = get_encode_fn();
    if (fn == nullptr) return false;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {inner * elem_bytes};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, type, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D bf16 tensor [outer, inner] (inner contiguous), box [box_outer, box_inner].
inline bool make_map(CUtensorMap* map, const void* base, uint64_t inner, uint64_t outer, uint32_t box_inner,
                     uint32_t box_outer, CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
    return make_map_typed(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, inner, outer, box_inner, box_outer, swizzle);
}

// Output map: [rows, cols] bf16, 32 x 32 blocks in the 64-byte swizzle pattern of the staging buffers.
inline bool make_out_map(CUtensorMap* map, const void* base, uint64_t cols, uint64_t rows) {
    return make_map(map, base, cols, rows, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B);
}

}  // namespace
}  // namespace moe

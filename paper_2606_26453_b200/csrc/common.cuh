// Shared declarations of the library's translation units (internal; not part of the C ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/moe_b200.h"

namespace moe {

typedef __nv_bfloat16 bf16;

// Device status word (one per device that loaded the library; lives in grouped_gemm.cu): kernels
// record MOE_ERR_TIMEOUT there when a bounded wait runs out.  Synchronises the device.
int read_and_clear_device_status(int* status_out);
int movement_read_and_clear_status(int* status_out);   // the data-movement kernels' word (movement.cu)
int mx_read_and_clear_status(int* status_out);         // the block-scaled FP8 kernels' word (mxfp8.cu)

// Number of SMs of the current device (cached per device ordinal).
int sm_count();

// CTA pairs the chip takes at once, one CTA per SM: what the rules of the dispatch count tiles against.  (The launches ask the device.)
constexpr int kChipPairs = 148 / 2;
// Rounds of tiles of `tile_rows` rows, times `feature_tiles`, for R rows of E experts, `at_once` of them at a time.  The host does not know
// the load: per expert the mean of the tiles of an even one and of one whose experts end anywhere in a tile.
inline double tile_rounds(long long R, int E, int tile_rows, long long feature_tiles, int at_once) {
    const double tiles = (double)R / E / tile_rows;
    return ceil(E * (ceil(tiles) + tiles + 0.5) / 2 * (double)feature_tiles / at_once);
}

// ---- programmatic dependent launch --------------------------------------------------------------
// The library's kernels are launched as programmatic dependents of whatever precedes them on the stream: their blocks may be
// placed, and may set up barriers, while the last blocks of the kernel before are still running.
// The rules that keep this equivalent to plain stream order:
//   - grid_dependency_wait() comes before a kernel's first access to global memory.  It returns once the kernels before have
//     completed and their writes are visible.  (rank_rows of the route-permute reads its INPUTS earlier: its predecessor, the
//     histogram or the scan kernel, lets it start only after its own wait and a fence, and it reads them past the L1; see the next rule but one.)
//   - grid_launch_dependents() comes after grid_dependency_wait(), so no more than one kernel is ever ahead of its turn and a
//     kernel that has started knows everything before its immediate predecessor to be complete.
//   - A weight gradient that a call launches right behind a data gradient on the same inputs does not depend on it.  Behind a
//     short one it runs beside it: no wait at its start (that it has started means that all before the data gradient is complete), the wait before
//     it lets ITS successor start, so that a kernel which has waited for it has waited for both.  Only a wait is documented to make
//     earlier kernels' writes visible, and this form reads without one.  What it reads was written before the data gradient; that
//     kernel's threads (it is told) have waited for those writes and fence (release_to_dependents) before any of them can trigger, so the writes
//     are performed at the scope of the device before the weight gradient can start, and its threads fence (acquire_unwaited) before they
//     read: nothing older comes out of an L1, by loads or by bulk copies.
//   - The GEMMs call it at the end of each warp's role.  One thread's call counts for its CTA, so the row-ragged bf16 kinds,
//     where one warp has no role, trigger right after set-up, and the CTAs of a GEMM that follows take each SM as it comes
//     free.  With the call behind the last barrier of the teardown steps of long GEMMs take longer, chip idle between steps:
//     8 experts of 4096 x 14336 11.78 -> 11.89 ms, 64 experts of 4096 x 1536 under a Zipf load 22.41 -> 22.73 ms, 128 of
//     2048 x 768 3.440 -> 3.448 ms.  (Presumably SMs that finish late get the CTAs with the fewest tiles.)
//   - Streaming kernels call it right behind their wait, except where there are many short blocks: the calls of a grid go
//     through one at a time, about 1 ns each, and a block that exits has triggered anyway (gather_sum_kernel, combine_bwd_kernel).
// Hides launch latency and set-up, 1.5-3 us at a kernel boundary: serving 32 tokens on 128 experts (six kernels) 167 -> 148 us,
// 100 tokens on FP8 weights 337 -> 261 us (both with what else changed since plain stream order); GEMM, streaming kernel,
// GEMM, streaming kernel on 1400 rows of 1024 44 -> 37 us.
// Kernels that read through read-only loads, which the compiler takes to be invariant, use the form whose result must be
// tested: the branch keeps such loads behind the wait.  (The GEMMs load their offsets through a plain pointer and everything
// else with bulk copies or behind a barrier; they take the plain form.)
// A small grid of 256-thread blocks: four on each of the chip's SMs.  (Asking the device for its SMs on every launch costs 0.1 us.)
constexpr unsigned kSmallGrid = 4 * 148;
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ bool grid_dependency_wait_tested() {
    uint32_t done;
    asm volatile("griddepcontrol.wait; mov.u32 %0, 1;" : "=r"(done) : : "memory");
    return done != 0;
}
// The two sides of a dependent that reads without waiting (see above).
__device__ __forceinline__ void release_to_dependents() { __threadfence(); }
__device__ __forceinline__ void acquire_unwaited() {
    __threadfence();
    asm volatile("fence.proxy.async.global;" ::: "memory");
}
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// `cluster`: CTAs per cluster.  `early` false: launched in plain stream order (the waits inside return at once).
template <typename... Params, typename... Args>
inline int launch_kernel(bool early, void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, unsigned cluster,
                         cudaStream_t s, const Args&... args) {
    cudaLaunchAttribute attr[2];
    unsigned n = 0;
    if (early) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster; attr[n].val.clusterDim.y = 1; attr[n++].val.clusterDim.z = 1;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(block); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cfg.attrs = attr; cfg.numAttrs = n;
    if (cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...) != cudaSuccess) {
        cudaGetLastError();
        return MOE_ERR_CUDA;
    }
    return MOE_OK;
}
template <typename... Params, typename... Args>
inline int launch_dependent(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, unsigned cluster, cudaStream_t s,
                            const Args&... args) {
    return launch_kernel(true, kernel, grid, block, smem, cluster, s, args...);
}
// Streaming kernels (256 threads, little or no shared memory).  Started early behind a GEMM their first blocks settle beside
// it, and that slows both: down dgrad and SwiGLU backward of 24576 x 1408 together (contraction of 256) 93 -> 102 us, of
// 131072 x 768 (contraction of 2048) 436 -> 463 us.  (Presumably such SMs keep the GEMM's split of their memory, with little
// L1 for loads in flight.)  So only small grids start early, which are over before that matters.
template <typename... Params, typename... Args>
inline int launch_streaming(void (*kernel)(Params...), unsigned grid, cudaStream_t s, const Args&... args) {
    return launch_kernel(grid <= kSmallGrid, kernel, grid, 256, 0, 1, s, args...);
}

// ---- data-movement kernels (movement.cu) ------------------------------------------------------
int launch_permute(const moe_dims_t& d, const bf16* x, const int32_t* topk_idx, bf16* x_perm,
                   int32_t* counts, int32_t* offsets, int32_t* row_to_pair, int32_t* pair_to_row,
                   void* workspace, cudaStream_t s);
size_t permute_workspace_bytes(const moe_dims_t& d);
int launch_permute_static_scratch(const moe_dims_t& d, const bf16* x, const int32_t* topk_idx, bf16* x_perm,
                                  int32_t* counts, int32_t* offsets, int32_t* row_to_pair, int32_t* pair_to_row,
                                  cudaStream_t s);
int launch_gather_sum(const moe_dims_t& d, const bf16* src_perm, const float* topk_w,
                      const int32_t* pair_to_row, bf16* dst, cudaStream_t s);  // topk_w may be NULL (unit weights)
int launch_combine_bwd(const moe_dims_t& d, const bf16* dy, const bf16* y_perm, const float* topk_w,
                       const int32_t* pair_to_row, bf16* dy_perm, float* dtopk_w, cudaStream_t s);
int launch_swiglu_bwd(const moe_dims_t& d, const bf16* dh_act, const bf16* gu, bf16* dgu, cudaStream_t s);

// ---- router (router.cu) ------------------------------------------------------------------------
int launch_router_topk(const moe_dims_t& d, const float* logits, int32_t* topk_idx, float* topk_w, cudaStream_t s);
int launch_router_topk_bwd(const moe_dims_t& d, const int32_t* topk_idx, const float* topk_w, const float* dtopk_w,
                           float* dlogits, cudaStream_t s);

// ---- grouped GEMMs (grouped_gemm.cu) -----------------------------------------------------------
int launch_gateup_fwd(const moe_dims_t& d, const bf16* x_perm, const bf16* w_gate, const bf16* w_up,
                      const int32_t* offsets, bf16* h_act, bf16* gu, cudaStream_t s);
int launch_down_fwd(const moe_dims_t& d, const bf16* h_act, const bf16* w_down, const int32_t* offsets,
                    bf16* y_perm, cudaStream_t s);
int launch_down_dgrad(const moe_dims_t& d, const bf16* dy_perm, const bf16* w_down, const int32_t* offsets,
                      bf16* dh_act, bool beside, cudaStream_t s);
int launch_down_wgrad(const moe_dims_t& d, const bf16* h_act, const bf16* dy_perm, const int32_t* offsets,
                      bf16* dw_down, bool beside, cudaStream_t s);   // beside: this right behind launch_down_dgrad, both with the same value; see above
int launch_down_dgrad_swiglu_bwd(const moe_dims_t& d, const bf16* dy_perm, const bf16* w_down, const bf16* gu,
                                 const int32_t* offsets, bf16* dgu, cudaStream_t s);
int launch_gateup_dgrad(const moe_dims_t& d, const bf16* dgu, const bf16* w_gate, const bf16* w_up,
                        const int32_t* offsets, bf16* dx_perm, bool beside, cudaStream_t s);
int launch_gateup_wgrad(const moe_dims_t& d, const bf16* x_perm, const bf16* dgu, const int32_t* offsets,
                        bf16* dw_gate, bf16* dw_up, bool beside, cudaStream_t s);

// ---- block-scaled FP8 down projection (mxfp8.cu) -------------------------------------------------
size_t mx_w_scale_single_bytes(int E, int n_feat, int k);   // weight scales in the single-CTA tiling
size_t mx_w_scale_bytes(int E, int n_feat, int k);          // both tilings, one after the other
int launch_mx_quantize_rows(long long rows, int n, const bf16* x, uint8_t* codes, uint8_t* scales, cudaStream_t s);
int launch_mx_quantize_w_transposed(int E, int k, int n, int n_total, int n_off, const bf16* w, uint8_t* codes_t, uint8_t* scales,
                                    cudaStream_t s);
int launch_mx_quantize_w_rows(int E, int n_feat, int k, int k_total, int k_off, const bf16* w, uint8_t* codes, uint8_t* scales,
                              cudaStream_t s);
long long mx_tokens_pitch(long long R, int E);            // columns of a token-quantised (transposed) operand
size_t mx_tokens_scale_bytes(long long R, int E, int n);
int launch_mx_quantize_tokens(long long R, int E, const bf16* x, long long ld, int col0, int n, const int32_t* offsets,
                              uint8_t* codes_t, uint8_t* scales, cudaStream_t s);
int launch_mx_wgrad(long long R, int E, int M, int N, const uint8_t* a_codes_t, const uint8_t* a_scales, const uint8_t* b_codes_t,
                    const uint8_t* b_scales, bf16* dw, cudaStream_t s);
int launch_mx_swiglu_quantize(long long rows, int I, const bf16* gu, bf16* h_act, uint8_t* codes, uint8_t* scales, cudaStream_t s);
int launch_mx_swiglu_bwd_quantize(long long rows, int I, const bf16* dh_act, const bf16* gu, bf16* dgu, uint8_t* codes,
                                  uint8_t* scales, cudaStream_t s);
int launch_mx_gemm(long long R, int E, int n_feat, int k, const uint8_t* a_codes, const uint8_t* a_scales, const uint8_t* b_codes,
                   const uint8_t* b_scales, const int32_t* offsets, bf16* out, cudaStream_t s);

}  // namespace moe

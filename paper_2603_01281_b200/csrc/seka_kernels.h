// Internal host-side launchers shared by the translation units of the library.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "seka_common.cuh"
#include "seka_prep.cuh"

namespace seka {

// Jobs that ride along with the preparation launch (see seka_prep.cuh).
struct PrepJobs {
    int n_items_blocks, n_conv_blocks;      // blocks for the item table (packed batches) and for the conversion (fp32 inputs)
    Sched sched;
    const int* cu;
    SteerIn steer;
    ItemRecord* items;
    int* item_count;
    ConvertArgs conv;
};

// The preparation of a forward without steering: `jobs` alone (nothing is launched if there are none).
seka_status launch_prep_plain(const PrepJobs& jobs, cudaStream_t st);

// Routing inside the preparation launch (Eq. 6); `sigma` null: the coefficients are given.
struct RouteArgs {
    const void* Q; int q_is_f32; const float* sigma; int k_route; int Hq; float* alpha_out;
};

// The preparation of a steered forward: edited keys of the tiles that hold a highlighted token into the side buffer
// X [T, Hkv, 2 d] (high | low parts), tile flags, steering bytes, and `jobs`.  K is the caller's tensor in its own dtype.
// With route.sigma set the coefficients are computed in the launch and written to route.alpha_out if that is not null.
seka_status launch_stage_keys(const seka_shape* s, const WorkspaceLayout& w, const void* K, const uint8_t* mask, const float* U,
                              const float* alpha, const float* gain, const uint8_t* head_enable, char* ws, const PrepJobs& jobs,
                              const RouteArgs& route, cudaStream_t st);

// Eq. 6 for every (sequence, KV head): the launch behind adaseka_route
seka_status launch_route(const seka_shape* s, const void* Q, const float* U, const float* sigma, int k_route,
                         float* alpha_out, cudaStream_t st);

// bf16 tensor [T, H, d] viewed as (d, H, T) for TMA: tiles of 64 x 1 x box_rows with the 128-byte swizzle.
bool make_tile_map(CUtensorMap* m, const void* base, int d, int H, long long T, int box_rows = 128);

// bf16 tensor [T, cols] for gathers of four rows x 64 columns at a time, 128-byte swizzle.
bool make_row_map(CUtensorMap* m, const void* base, int cols, long long T);

seka_status validate_shape(const seka_shape* s);

// Number of SMs of the current device (looked up once per device, thread-safe).
bool device_info(int* n_sm);

// Launch whose status is that of the launch alone.  With `pdl` it may be placed while its predecessor in the stream drains
// (the kernel begins with pdl_wait).  `cluster`: CTAs of a cluster along x.
template <typename... P, typename... A>
static inline seka_status launch_cluster(bool pdl, unsigned cluster, void (*kern)(P...), dim3 grid, unsigned threads, size_t smem,
                                         cudaStream_t st, const A&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute at[2];
    unsigned n = 0;
    if (pdl) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = cluster; at[n].val.clusterDim.y = 1; at[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = at; cfg.numAttrs = n;
    if (cudaLaunchKernelEx(&cfg, kern, args...) != cudaSuccess) return SEKA_ERR_CUDA;
    ++g_launches;
    return SEKA_OK;
}
template <typename... P, typename... A>
static inline seka_status launch_kernel(bool pdl, void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st,
                                        const A&... args) {
    return launch_cluster(pdl, 1u, kern, grid, threads, smem, st, args...);
}

}  // namespace seka

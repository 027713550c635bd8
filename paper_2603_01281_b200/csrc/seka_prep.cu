// Preparation of a forward without steering: what it needs beside the attention kernel (item table of a packed batch, bf16
// copies of fp32 inputs), in one launch.  With steering the same jobs run in blocks of the key-editing launch (seka_edit.cu).
#include "seka_kernels.h"

namespace seka {

__global__ void __launch_bounds__(PREP_THREADS)
prep_plain_kernel(const __grid_constant__ PrepJobs jobs) {
    pdl_wait();
    pdl_release();
    if ((int)blockIdx.x < jobs.n_items_blocks)
        items_block(jobs.sched, jobs.cu, jobs.steer, jobs.items, jobs.item_count, blockIdx.x);
    else
        convert_block(jobs.conv, blockIdx.x - jobs.n_items_blocks, jobs.n_conv_blocks);
}

seka_status launch_prep_plain(const PrepJobs& jobs, cudaStream_t st) {
    const unsigned grid = (unsigned)(jobs.n_items_blocks + jobs.n_conv_blocks);
    if (grid == 0) return SEKA_OK;
    return launch_kernel(true, prep_plain_kernel, grid, PREP_THREADS, 0, st, jobs);
}

}  // namespace seka

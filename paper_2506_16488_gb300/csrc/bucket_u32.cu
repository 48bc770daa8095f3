// The bucketed kernel over adjacency blocks, for 32-bit tentative distances.
#include "bucket_core.cuh"

namespace ppsp {

ppsp_status launch_bucket_u32(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream) {
    return bucket_launch<u32, BK_CTAS>(a, block_threads, grid, stream);
}

ppsp_status occupancy_bucket_u32(int block_threads, u32 ring_cap, int* bpsm) {
    return bucket_occ<u32, BK_CTAS>(block_threads, ring_cap, bpsm);
}

}  // namespace ppsp

// The bucketed kernel over adjacency blocks, for 64-bit tentative distances, with teams of several CTAs.
#include "bucket_core.cuh"

namespace ppsp {

ppsp_status launch_bucket_u64_teams(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream) {
    return bucket_launch<u64, BK_TEAMS>(a, block_threads, grid, stream);
}

ppsp_status occupancy_bucket_u64_teams(int block_threads, u32 ring_cap, int* bpsm) {
    return bucket_occ<u64, BK_TEAMS>(block_threads, ring_cap, bpsm);
}

}  // namespace ppsp

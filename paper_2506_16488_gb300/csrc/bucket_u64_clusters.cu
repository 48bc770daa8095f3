// The bucketed kernel over adjacency blocks, for 64-bit tentative distances, on clusters.
#include "bucket_core.cuh"

namespace ppsp {

ppsp_status launch_bucket_u64_clusters(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream) {
    return bucket_launch<u64, BK_CLUSTERS>(a, block_threads, grid, stream);
}

ppsp_status resident_bucket_u64_clusters(int block_threads, u32 ring_cap, u32 cluster, int* clusters) {
    return bucket_clusters<u64>(block_threads, ring_cap, cluster, clusters);
}

}  // namespace ppsp

// Engine dispatch by distance width, and the small kernels of a plan run
// (potential evaluation, result scatter).
#include <map>
#include <mutex>
#include <tuple>

#include "engine_core.cuh"

namespace ppsp {

// instantiated in engine_{u32,u64}{,_local}.cu
ppsp_status launch_engine_u32(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream);
ppsp_status launch_engine_u64(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream);
ppsp_status launch_engine_u32_local(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream);
ppsp_status launch_engine_u64_local(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream);
ppsp_status engine_occupancy_u32(int block_threads, u32 ring_cap, int* bpsm);
ppsp_status engine_occupancy_u64(int block_threads, u32 ring_cap, int* bpsm);
ppsp_status engine_occupancy_u32_local(int block_threads, u32 ring_cap, int* bpsm);
ppsp_status engine_occupancy_u64_local(int block_threads, u32 ring_cap, int* bpsm);
// instantiated in bucket_{u32,u64}{,_teams,_clusters}.cu
ppsp_status launch_bucket_u32(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream);
ppsp_status launch_bucket_u64(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream);
ppsp_status launch_bucket_u32_teams(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream);
ppsp_status launch_bucket_u64_teams(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream);
ppsp_status launch_bucket_u32_clusters(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream);
ppsp_status launch_bucket_u64_clusters(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream);
ppsp_status resident_bucket_u32_clusters(int block_threads, u32 ring_cap, u32 cluster, int* clusters);
ppsp_status resident_bucket_u64_clusters(int block_threads, u32 ring_cap, u32 cluster, int* clusters);
ppsp_status occupancy_bucket_u32(int block_threads, u32 ring_cap, int* bpsm);
ppsp_status occupancy_bucket_u64(int block_threads, u32 ring_cap, int* bpsm);
ppsp_status occupancy_bucket_u32_teams(int block_threads, u32 ring_cap, int* bpsm);
ppsp_status occupancy_bucket_u64_teams(int block_threads, u32 ring_cap, int* bpsm);

ppsp_status launch_engine(const EngineArgs& a, int dist_bits, int block_threads, u32 grid,
                          cudaStream_t stream, EngineKind kind) {
    const bool w32 = dist_bits == 32;
    if (kind == ENGINE_BUCKET && a.long_ctas && a.part == 0) {
        // The longest groups on more threads each, the rest beside them.  Neither
        // launch waits for the other's groups, so only the time depends on their
        // running at once.
        if (a.long_ctas >= grid || a.cluster < 1 || a.long_ctas % a.cluster) return PPSP_ERR_INVALID_ARG;
        EngineArgs one = a, two = a;
        one.part = 1;
        one.ring_cap = a.long_cap;
        two.part = 2;
        two.team0 = a.long_ctas / a.cluster;
        const ppsp_status st = launch_engine(one, dist_bits, 1024, a.long_ctas, stream,
                                             a.cluster > 1 ? ENGINE_BUCKET_CLUSTERS : ENGINE_BUCKET);
        return st == PPSP_OK ? launch_engine(two, dist_bits, block_threads, grid - a.long_ctas, stream, ENGINE_BUCKET)
                             : st;
    }
    if (kind == ENGINE_BUCKET)
        return w32 ? launch_bucket_u32(a, block_threads, grid, stream) : launch_bucket_u64(a, block_threads, grid, stream);
    if (kind == ENGINE_BUCKET_CLUSTERS)
        return w32 ? launch_bucket_u32_clusters(a, block_threads, grid, stream)
                   : launch_bucket_u64_clusters(a, block_threads, grid, stream);
    if (kind == ENGINE_BUCKET_TEAMS)
        return w32 ? launch_bucket_u32_teams(a, block_threads, grid, stream)
                   : launch_bucket_u64_teams(a, block_threads, grid, stream);
    if (kind == ENGINE_LOCAL)
        return w32 ? launch_engine_u32_local(a, block_threads, grid, stream)
                   : launch_engine_u64_local(a, block_threads, grid, stream);
    return w32 ? launch_engine_u32(a, block_threads, grid, stream) : launch_engine_u64(a, block_threads, grid, stream);
}

// Occupancy answers, kept per device and configuration (a query to the driver
// costs more than the rest of a small plan).
namespace {
struct OccCache {
    std::mutex mu;
    std::map<std::tuple<int, int, int, int, u32, u32>, int> got;
} g_occ;

template <typename F>
ppsp_status occ_cached(int kind, int dist_bits, int block, u32 cap, u32 cluster, int* out, F ask) {
    int dev = 0;
    PPSP_CUDA_TRY(cudaGetDevice(&dev));
    const auto key = std::make_tuple(dev, kind, dist_bits, block, cap, cluster);
    std::lock_guard<std::mutex> lk(g_occ.mu);
    auto it = g_occ.got.find(key);
    if (it == g_occ.got.end()) {
        int v = 0;
        const ppsp_status st = ask(dev, &v);
        if (st != PPSP_OK) return st;
        it = g_occ.got.emplace(key, v).first;
    }
    *out = it->second;
    return PPSP_OK;
}
}  // namespace

ppsp_status engine_occupancy(int dist_bits, int block_threads, int* blocks_per_sm, int* sms, EngineKind kind,
                             u32 ring_cap) {
    ppsp_status st = occ_cached(-1, 0, 0, 0, 0, sms, [](int dev, int* v) {
        PPSP_CUDA_TRY(cudaDeviceGetAttribute(v, cudaDevAttrMultiProcessorCount, dev));
        return PPSP_OK;
    });
    if (st != PPSP_OK) return st;
    const bool w32 = dist_bits == 32;
    return occ_cached(kind, dist_bits, block_threads, ring_cap, 0, blocks_per_sm, [=](int, int* v) {
        switch (kind) {
            case ENGINE_BUCKET:
                return w32 ? occupancy_bucket_u32(block_threads, ring_cap, v)
                           : occupancy_bucket_u64(block_threads, ring_cap, v);
            case ENGINE_BUCKET_TEAMS:
                return w32 ? occupancy_bucket_u32_teams(block_threads, ring_cap, v)
                           : occupancy_bucket_u64_teams(block_threads, ring_cap, v);
            case ENGINE_LOCAL:
                return w32 ? engine_occupancy_u32_local(block_threads, ring_cap, v)
                           : engine_occupancy_u64_local(block_threads, ring_cap, v);
            default:
                return w32 ? engine_occupancy_u32(block_threads, ring_cap, v)
                           : engine_occupancy_u64(block_threads, ring_cap, v);
        }
    });
}

ppsp_status engine_clusters(int dist_bits, int block_threads, u32 ring_cap, u32 cluster, int* clusters) {
    return occ_cached(ENGINE_BUCKET_CLUSTERS, dist_bits, block_threads, ring_cap, cluster, clusters,
                      [=](int, int* v) {
                          return dist_bits == 32 ? resident_bucket_u32_clusters(block_threads, ring_cap, cluster, v)
                                                 : resident_bucket_u64_clusters(block_threads, ring_cap, cluster, v);
                      });
}

// ---- adjacency blocks: one thread per record of a block; the thread of a
// fourth record that continues writes the rest of the row ----
__global__ void fill_blocks_kernel(const u32* off, const uint2* edges, const int4* edges_pc, const u32* more, u32 n,
                                   uint2* blk8, int4* blk16) {
    const u64 k = (u64)blockIdx.x * blockDim.x + threadIdx.x;
    const u64 v = k >> 2;
    if (v >= n) return;
    const u32 b0 = off[v], deg = off[v + 1] - b0, q = (u32)(k & 3);
    const bool cont = deg > 4 && q == 3;
    auto put = [&](u64 at, u32 e) {  // edge e, or an unused record
        const uint2 none = make_uint2(BLK_NONE, 0u);
        uint2 r = e < b0 + deg ? edges[e] : none;
        int4 p = (blk16 && e < b0 + deg) ? edges_pc[e] : make_int4(0, 0, 0, 0);
        if (e < b0 + deg && off[r.x + 1] - off[r.x] > 4) r.x |= 1u << 31;
        if (blk8) blk8[at] = r;
        if (blk16) blk16[at] = make_int4((int)r.x, (int)r.y, p.z, p.w);
    };
    if (!cont) {
        put(k, b0 + q);
        return;
    }
    const u32 at = more[v];
    if (blk8) blk8[k] = make_uint2(BLK_MORE, at);
    if (blk16) blk16[k] = make_int4((int)BLK_MORE, (int)at, 0, 0);
    // deg - 3 records, padded to a multiple of four
    for (u32 j = 0; j < (deg & ~3u); ++j) put((u64)at + j, b0 + 3 + j);
}

ppsp_status launch_fill_blocks(const u32* off, const uint2* edges, const int4* edges_pc, const u32* more, u32 n,
                               uint2* blk8, int4* blk16) {
    const u64 blocks = ((u64)n * 4 + 255) / 256;
    fill_blocks_kernel<<<(u32)blocks, 256>>>(off, edges, edges_pc, more, n, blk8, blk16);
    PPSP_CUDA_TRY(cudaGetLastError());
    return PPSP_OK;
}

// ---- potential evaluation (for checks against the oracle) ----
__global__ void potential_eval_kernel(GraphDev g, u32 anchor, const u32* verts, u64 count, i64* out) {
    u64 k = (u64)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= count) return;
    u32 v = verts[k];
    out[k] = (v < g.n) ? pot_h(g.pc[anchor], g.pc[v], g.pot_shift) : -1;
}

ppsp_status launch_potential_eval(const GraphDev& g, u32 anchor, const u32* d_verts, u64 count,
                                  i64* d_out, cudaStream_t stream) {
    if (count == 0) return PPSP_OK;
    u32 blocks = (u32)((count + 255) / 256);
    potential_eval_kernel<<<blocks, 256, 0, stream>>>(g, anchor, d_verts, count, d_out);
    PPSP_CUDA_TRY(cudaGetLastError());
    return PPSP_OK;
}

__global__ void scatter_kernel(const u32* map, const u64* mu, u64 k, u64* out) {
    u64 q = (u64)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= k) return;
    u32 m = map[q];
    out[q] = (m == NONE) ? 0ull : mu[m];
}

ppsp_status launch_scatter(const u32* d_map, const u64* d_mu, u64 k, u64* d_out, cudaStream_t s) {
    if (k == 0) return PPSP_OK;
    u32 blocks = (u32)((k + 255) / 256);
    scatter_kernel<<<blocks, 256, 0, s>>>(d_map, d_mu, k, d_out);
    PPSP_CUDA_TRY(cudaGetLastError());
    return PPSP_OK;
}

}  // namespace ppsp


// Batch planning: query graph (Sec. 4.1), groups, team schedule, launches.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <numeric>
#include <unordered_map>
#include <unordered_set>

#include "graph_impl.h"
#include "mlp_internal.h"

using namespace ppsp;

struct ppsp_plan {
    ppsp_graph* g = nullptr;
    ppsp_options opt{};
    cudaStream_t stream = nullptr;
    u64 k = 0;
    int dist_bits = 32;
    int block = 512;
    EngineKind kind = ENGINE_GENERAL;
    bool memo = false;                 // slots keep memoized potential terms (Sec. 5)
    u32 grid = 0;
    std::vector<GroupDev> groups;
    std::vector<SearchDev> searches;
    std::vector<PartnerDev> partners;
    std::vector<QEdgeDev> qedges;
    std::vector<u32> map;              // input query -> global query edge, NONE for s == t
    std::vector<std::pair<u32, u32>> qedge_ends;  // global query edge -> (s, t) vertices
    std::vector<u32> team_first, team_size, team_queue, cta_team;
    std::vector<u32> queue_items[MAX_QUEUES];
    std::vector<Slot*> slots;
    void* d_arena = nullptr;
    size_t arena_bytes = 0;
    char* d_runstate = nullptr;
    size_t runstate_bytes = 0;
    u32* d_map = nullptr;
    EngineArgs args{};
    bool launched = false;
    bool host_call = false;     // one call from host pairs to host answers: the arena is the graph's workspace
    size_t back_at = 0, back_bytes = 0;  // arena range with the error word, the counters and mu
    // learned Delta: per-group features (log2(1 + raw)) and the model used
    std::vector<float> feats;
    float* d_feats = nullptr;
    ppsp_delta_model* model = nullptr;
    u64 delta_default = 1;
    // paths (ppsp_query / ppsp_batch with want_paths)
    bool paths = false;
    std::vector<u64> path_off;  // [qedges + 1]
    void* d_paths = nullptr;    // path buffer, offsets, lengths, meeting vertices
    u32* d_meet = nullptr;
    // CUDA-graph replay of plan_run (per output pointer)
    cudaGraphExec_t gexec = nullptr;
    u64* gexec_out = nullptr;
    bool graph_failed = false;
    bool last_used_graph = false;
};

namespace {

struct UF {
    std::vector<u32> p;
    explicit UF(u32 n) : p(n) { std::iota(p.begin(), p.end(), 0u); }
    u32 find(u32 x) {
        while (p[x] != x) x = p[x] = p[p[x]];
        return x;
    }
    void join(u32 a, u32 b) {
        a = find(a);
        b = find(b);
        if (a != b) p[std::max(a, b)] = std::min(a, b);
    }
};

// Minimum vertex cover of a graph of at most 32 vertices given as adjacency
// bit masks, by branch and bound: take the vertex v of largest uncovered
// degree and branch on "v in the cover" / "all uncovered neighbours of v in
// the cover"; a greedy maximal matching of the uncovered edges bounds the
// rest from below (every matching edge needs its own cover vertex), and once
// no vertex has two uncovered edges the remaining edges form a matching.
void vc_exact(const std::vector<u32>& adj, u32 cover, u32 size, u32& best_size, u32& best) {
    if (size >= best_size) return;
    const u32 nv = (u32)adj.size();
    u32 v = 0, maxd = 0;
    for (u32 u = 0; u < nv; ++u) {
        if (cover >> u & 1u) continue;
        const u32 d = (u32)__builtin_popcount(adj[u] & ~cover);
        if (d > maxd) {
            maxd = d;
            v = u;
        }
    }
    if (maxd <= 1) {
        u32 c = cover, sz = size;
        for (u32 u = 0; u < nv; ++u)
            if (!(c >> u & 1u) && (adj[u] & ~c)) {
                c |= 1u << u;
                ++sz;
            }
        if (sz < best_size) {
            best_size = sz;
            best = c;
        }
        return;
    }
    u32 m = cover, lb = 0;
    for (u32 u = 0; u < nv; ++u) {
        if (m >> u & 1u) continue;
        const u32 w = adj[u] & ~m;
        if (w) {
            m |= (1u << u) | (w & (0u - w));
            ++lb;
        }
    }
    if (size + lb >= best_size) return;
    vc_exact(adj, cover | (1u << v), size + 1, best_size, best);
    const u32 nb = adj[v] & ~cover;
    vc_exact(adj, cover | nb, size + (u32)__builtin_popcount(nb), best_size, best);
}

// Vertex cover of the query graph (Sec. 4.3): exact for components of at most
// 32 vertices, greedy by uncovered degree otherwise.  Returns in[v] for the
// local vertex ids 0..nv-1.
std::vector<char> vertex_cover(u32 nv, const std::vector<std::pair<u32, u32>>& E) {
    std::vector<u32> comp(nv);
    std::iota(comp.begin(), comp.end(), 0u);
    std::function<u32(u32)> find = [&](u32 x) { return comp[x] == x ? x : comp[x] = find(comp[x]); };
    for (auto& e : E) comp[find(e.first)] = find(e.second);
    std::unordered_map<u32, std::vector<u32>> cv;
    std::unordered_map<u32, std::vector<std::pair<u32, u32>>> ce;
    for (u32 v = 0; v < nv; ++v) cv[find(v)].push_back(v);
    for (auto& e : E) ce[find(e.first)].push_back(e);
    std::vector<char> in(nv, 0);
    for (auto& kv : cv) {
        auto& verts = kv.second;
        auto& edges = ce[kv.first];
        if (edges.empty()) continue;
        if (verts.size() <= 32) {
            std::unordered_map<u32, u32> loc;
            for (u32 i = 0; i < verts.size(); ++i) loc[verts[i]] = i;
            std::vector<u32> adj(verts.size(), 0u);
            for (auto& e : edges) {
                const u32 x = loc[e.first], y = loc[e.second];
                adj[x] |= 1u << y;
                adj[y] |= 1u << x;
            }
            u32 best = (verts.size() == 32) ? ~0u : ((1u << verts.size()) - 1u), best_size = (u32)verts.size();
            vc_exact(adj, 0u, 0, best_size, best);
            for (u32 i = 0; i < verts.size(); ++i) in[verts[i]] = (char)(best >> i & 1u);
        } else {
            std::vector<char> covered(edges.size(), 0);
            size_t left = edges.size();
            while (left) {
                std::unordered_map<u32, u32> deg;
                for (size_t k = 0; k < edges.size(); ++k)
                    if (!covered[k]) {
                        ++deg[edges[k].first];
                        ++deg[edges[k].second];
                    }
                u32 pick = 0, pd = 0;
                for (auto& d : deg)
                    if (d.second > pd || (d.second == pd && d.first < pick)) {
                        pick = d.first;
                        pd = d.second;
                    }
                in[pick] = 1;
                for (size_t k = 0; k < edges.size(); ++k)
                    if (!covered[k] && (edges[k].first == pick || edges[k].second == pick)) {
                        covered[k] = 1;
                        --left;
                    }
            }
        }
    }
    return in;
}

// Minimum vertex cover of a bipartite graph (left 0..nl-1, right
// 0..nr-1): a maximum matching by augmenting paths, then Konig's
// construction (left vertices not reachable by alternating paths from free
// left vertices, right vertices reachable).  Returns cover flags.
void bipartite_cover(u32 nl, u32 nr, const std::vector<std::pair<u32, u32>>& E, std::vector<char>& inl,
                     std::vector<char>& inr) {
    std::vector<std::vector<u32>> adjl(nl);
    for (auto& e : E) adjl[e.first].push_back(e.second);
    std::vector<u32> ml(nl, NONE), mr(nr, NONE);
    std::vector<u32> seen(nr, NONE);
    // iterative augmenting-path search from left vertex r0 (stamp = r0)
    auto augment = [&](u32 r0) {
        std::vector<std::pair<u32, u32>> st;  // (left vertex, next edge index)
        std::vector<u32> via;                 // right vertex taken from each frame
        st.emplace_back(r0, 0);
        while (!st.empty()) {
            auto& [x, k] = st.back();
            if (k == adjl[x].size()) {
                st.pop_back();
                if (!via.empty()) via.pop_back();
                continue;
            }
            const u32 y = adjl[x][k++];
            if (seen[y] == r0) continue;
            seen[y] = r0;
            if (mr[y] == NONE) {
                // flip the path: frames hold left vertices, via the right ones
                via.push_back(y);
                for (size_t f = st.size(); f-- > 0;) {
                    const u32 lx = st[f].first, ry = via[f];
                    ml[lx] = ry;
                    mr[ry] = lx;
                }
                return true;
            }
            via.push_back(y);
            st.emplace_back(mr[y], 0);
        }
        return false;
    };
    for (u32 x = 0; x < nl; ++x) augment(x);
    // alternating reachability from free left vertices
    std::vector<char> zl(nl, 0), zr(nr, 0);
    std::vector<u32> queue;
    for (u32 x = 0; x < nl; ++x)
        if (ml[x] == NONE) {
            zl[x] = 1;
            queue.push_back(x);
        }
    for (size_t h = 0; h < queue.size(); ++h) {
        const u32 x = queue[h];
        for (u32 y : adjl[x])
            if (!zr[y] && ml[x] != y) {
                zr[y] = 1;
                const u32 x2 = mr[y];
                if (x2 != NONE && !zl[x2]) {
                    zl[x2] = 1;
                    queue.push_back(x2);
                }
            }
    }
    inl.assign(nl, 0);
    inr.assign(nr, 0);
    for (u32 x = 0; x < nl; ++x) inl[x] = zl[x] ? 0 : 1;
    for (u32 y = 0; y < nr; ++y) inr[y] = zr[y] ? 1 : 0;
}

// Search that answers each query (s, t) of an SSSP-based batch (Sec. 4.3),
// as (vertex, direction): Plain-SSSP searches forward from s; VC-SSSP from an
// endpoint in a vertex cover of G_q: on an undirected graph (direction 0)
// exact up to 32 vertices per component and greedy above; on a directed
// graph G_q is bipartite (sources, targets: Sec. 4.4) and its minimum cover
// comes from a maximum matching (Konig); a target in the cover searches
// backward (direction 1) over the transpose.
struct SrcDir {
    u32 v;
    u32 dir;
};
std::vector<SrcDir> sssp_sources(int strategy, bool directed, const std::vector<std::pair<u32, u32>>& uq) {
    const u32 U = (u32)uq.size();
    std::vector<SrcDir> src(U);
    if (strategy != PPSP_BATCH_VC) {
        for (u32 u = 0; u < U; ++u) src[u] = {uq[u].first, 0};
        return src;
    }
    if (directed) {
        std::unordered_map<u32, u32> lid, rid;
        std::vector<std::pair<u32, u32>> E(U);
        for (u32 u = 0; u < U; ++u)
            E[u] = {lid.emplace(uq[u].first, (u32)lid.size()).first->second,
                    rid.emplace(uq[u].second, (u32)rid.size()).first->second};
        std::vector<char> inl, inr;
        bipartite_cover((u32)lid.size(), (u32)rid.size(), E, inl, inr);
        for (u32 u = 0; u < U; ++u)
            src[u] = inl[E[u].first] ? SrcDir{uq[u].first, 0} : SrcDir{uq[u].second, 1};
        return src;
    }
    std::unordered_map<u32, u32> vid;
    std::vector<u32> verts;
    auto get = [&](u32 v) {
        auto it = vid.find(v);
        if (it != vid.end()) return it->second;
        vid.emplace(v, (u32)verts.size());
        verts.push_back(v);
        return (u32)verts.size() - 1;
    };
    std::vector<std::pair<u32, u32>> le(U);
    for (u32 u = 0; u < U; ++u) le[u] = {get(uq[u].first), get(uq[u].second)};
    const std::vector<char> in = vertex_cover((u32)verts.size(), le);
    for (u32 u = 0; u < U; ++u) src[u] = {in[le[u].first] ? uq[u].first : uq[u].second, 0};
    return src;
}

// Time of a group of 512 threads beside another one on the SM, over that of
// 1,024 threads alone, for all groups and the longest: 1,000 BiD-A* queries on
// the 1024^2 road graph 1.47, the 32 longest of them 1.59; one-directional A*
// on 500^2 1.35 and 1.40.
constexpr double GROUP_512 = 1.45, LONG_512 = 1.6;

// Bucketed kernel: shared-memory entries per bucket.  The ring (64 buckets of
// 8- or 16-byte entries) takes 128 KB of an SM, whatever the CTAs' size.
u32 bucket_cap(int block, int dist_bits) { return (u32)block / 4 / (dist_bits == 64 ? 2 : 1); }
// The same from the ring_entries option: at most what fits a CTA's shared memory.
u32 bucket_cap(u32 ring_entries, int block, int dist_bits) {
    if (!ring_entries) return bucket_cap(block, dist_bits);
    return std::min(ring_entries, dist_bits == 64 ? BK_RING_MAX_64 : BK_RING_MAX_32);
}

// Estimated device time (us) of a group of one or two searches on the bucketed
// kernel with clusters of `cl` CTAs of 1,024 threads.  H: the queries' largest
// heuristic distance in mean edge weights.  A step of e entries takes about
// 2.2 + 0.0105 e us on one CTA, and a cluster splits the entries and pays 2 us
// for its barrier and the others' states; a group takes about 1.2 H steps of
// c H entries (road-like graphs of 512^2 to 4096^2, six random pairs or a
// 64-leaf star each: BiD-A* c = 0.25 to 0.36, BiDS 1.05, ET and single-source
// 2.1 to 2.4).  Searches with a potential take more steps per H the longer the
// query (BiD-A*: 1.29 at a mean H of 483, 1.5 at 1974).
// busy: what a cluster's entry costs more, over one CTA's.
// threads: of a CTA; an entry takes LONG_512 times as long with half of them.
double bucket_group_us(u32 mode, bool pot, double H, double n, u32 cl, double busy = 0.0, int threads = 1024) {
    const double c = mode == GM_BIDIR ? (pot ? 0.3 : 1.05) : mode == GM_ASTAR ? 0.5 : 2.2;
    const double steps = 1.2 * H * (pot ? std::pow(std::max(H, 1.0) / 500.0, 0.15) : 1.0) + 20.0;
    const double entries = std::min(c * H, 2.0 * n / steps);
    const double entry = 0.0105 * std::pow(LONG_512, std::log2(1024.0 / threads));
    return steps * (2.2 + (cl > 1 ? 2.0 : 0.0) + entry * entries * (1.0 / cl + (cl > 1 ? busy : 0.0)));
}

// What a cluster's entry costs more while the other SMs are busy, over one
// CTA's entry: 256 BiD-A* queries on the 4096^2 graph, the longest on four CTAs
// 83 ms where one takes 105.
constexpr double CLUSTER_BUSY = 0.3;
// A group takes up to this much longer than estimated.
constexpr double LONG_SPREAD = 1.3;

// Whether the longest BiD-A* pairs of a batch should start on more threads than
// the rest, in a launch of their own, so that they do not outlast it.  Measured
// in one launch / two: 1,000 queries on the 1024^2 road graph (two groups per
// SM; the longest 15.6 ms, all together 11.8) 15.6 / 12.7 ms; 40, 150, 300, 700
// on 2048^2 23.4, 32.3, 32.7, 60.4 / 16.7, 20.5, 24.1, 36.8; 256 with 64-bit
// distances on 4096^2 105 / 82.  Not for other searches, whose estimates are
// too rough and whose clusters slow one another more: 160 and 300 BiDS pairs
// on 1024^2 10.2, 10.5 / 12.2, 12.9.
// us: estimated times by CTAs per group (1, 2, 4, 8; 1,024 threads each),
// longest first; per_sm: groups per SM of the rest; best: the estimate without.
// Each count q of longest groups is tried with each size: the time is at least
// that of its longest group, that of the rest's longest, and everything over
// the SMs.
struct LongGroups {
    u32 groups = 0, cl = 1, teams = 0;
};
LongGroups long_groups(const std::vector<double> us[4], const u32 max_teams[4], u32 sms, u32 per_sm, double best) {
    LongGroups r;
    const double share = per_sm > 1 ? GROUP_512 : 1.0, tail = LONG_SPREAD * (per_sm > 1 ? LONG_512 : 1.0);
    const u32 ng = (u32)us[0].size();
    double all = 0;
    for (double x : us[0]) all += x * share / per_sm;
    best *= 0.95;
    for (u32 c = per_sm > 1 ? 0 : 1; c < 4; ++c) {
        if (us[c].empty()) continue;
        double head = 0, longest = 0, rest = all;  // the longest groups' times, SM time of the rest
        for (u32 q = 1; q < ng; ++q) {
            head += us[c][q - 1];
            longest = std::max(longest, us[c][q - 1]);
            rest -= us[0][q - 1] * share / per_sm;
            const u32 teams = std::min({q, max_teams[c], (3 * sms / 4) >> c});
            if (teams == 0) break;
            const double t = std::max({longest, head / teams, us[0][q] * tail, (head * (1u << c) + rest) / sms});
            if (t < best) {
                best = t;
                r = {q, 1u << c, teams};
            }
        }
    }
    return r;
}

// Stepping increment of an A* group when no model is attached (mean edge
// weight over this): along the shortest path the keys barely grow, so the
// threshold runs ahead by one increment per hop, and a long path wants a small
// one.  H: heuristic distance in mean edge weights.  One-directional A*, six
// random pairs, w/4, w/8, w/16: 512^2 (H about 265) 12.2, 6.6, 11.3 ms; 1024^2
// 57, 13.7, 16.1; 2048^2 1037, 224, 60.  BiD-A*, 1,000 pairs on 1024^2, w/4,
// w/8, w/16, w/32: 139, 25.9, 16.2, 19.9 ms.  On graphs that grow faster than the
// plane paths have few hops and one mean weight stays, but for one-directional
// A* on one CTA per group (random graph of 2^20 vertices with coordinates, one
// mean weight / this: A* 8 queries one at a time 4.7 / 7.5 ms, 24 pairs 12.9 /
// 25.9, 200 906 / 181; BiD-A* 1,000 pairs 2.0 / 2.2).
double astar_divisor(bool bidir, double H) {
    return bidir ? std::min(32.0, std::max(8.0, H / 32.0)) : std::min(32.0, std::max(6.0, H / 64.0));
}

// Whether a plan takes the kernels over adjacency blocks (on a graph that has
// them).  Where neighbourhoods grow as in the plane, always.  Elsewhere the steps
// of a search have very many entries, which outgrow a CTA's buckets and their
// overflow regions, so large graphs, graphs with long rows and few groups, which
// have many CTAs each on the queue path, keep the other kernels.  Measured, queue
// path or run_local / this kernel: one query at a time, ET on a random graph of
// 2^20 vertices (average degree 5.5) 1.3 / 132 ms, BiDS on RMAT-20 with edge
// factor 3 6.2 / 165, BiDS on a 100^3 grid 1.4 / 61; 200 at once: ET on random
// graphs of 2^15, 2^16, 2^17, 2^20 vertices 21, 68, 101, 1,490 / 2.5, 15, 37,
// 3,860 ms, BiDS on RMAT-13 and -15 with edge factor 3 1.4, 5.8 / 1.9, 10.2.
// Bidirectional searches of a random graph settle about sqrt(n) vertices and
// are short whatever its size: 24 BiDS pairs on 2^15, 2^18, 2^20 vertices 0.22,
// 0.32, 0.49 / 0.09, 0.17, 0.32; 1,000 pairs on 2^17 vertices 1.1 / 2.7.
// ctas: CTAs that run everything at once; one: one CTA per group.
bool blocks_pay(const ppsp_graph* g, bool all_bidir, bool one, bool pairs_only, u64 ctas, u32 sms) {
    if (g->growth == GROWTH_PLANE || g->n <= BLOCK_SMALL_N) return true;
    if (g->info.deg_max > BLOCK_MAX_ROW) return false;
    return (g->growth == GROWTH_RANDOM && all_bidir && ctas <= sms) || (one && pairs_only && g->n <= (1u << 16));
}

// AUTO strategy: smallest number of targets that makes a source's queries
// one multi-target search (ET / A* modes).
constexpr u32 AUTO_MIN_TARGETS = 4;

// AUTO strategy, per connected component of G_q with nv vertices, ne edges
// and a vertex cover of `cover` vertices.  With BiD-A* potentials a pair
// search settles far fewer vertices than an unpruned or shared search (the
// potential is only exact for isolated pairs, so shared searches lose it):
// components run as independent pairs unless one vertex covers the whole
// component (a star), whose one search from the centre answers every query.
// Without potentials, a cover of at most a quarter of the vertices runs as
// VC-SSSP (stars, forks), the rest as Multi-BiDS (Sec. 4.2 / 4.3).  On a
// dense low-diameter graph (average degree at least AUTO_DENSE_DEG, the
// social-graph shape) every component, an isolated pair too, runs as
// VC-SSSP: there a search that stops at its last target beats the
// bidirectional searches (measured on RMAT-22: 1.6 s against 3.7 s for the
// same batch, Sec. 4.3 notes the same trend for social graphs).
constexpr double AUTO_DENSE_DEG = 8.0;
int auto_component(bool pot_pairs, bool dense, u32 nv, u32 ne, u32 cover) {
    if (pot_pairs) return (cover == 1 && ne >= AUTO_MIN_TARGETS) ? PPSP_BATCH_VC : PPSP_BATCH_PLAIN_STAR;
    if (dense) return PPSP_BATCH_VC;
    return (4u * cover <= nv) ? PPSP_BATCH_VC : PPSP_BATCH_MULTI;
}

u32 ceil_log2(u32 x) {
    u32 s = 0;
    while ((1u << s) < x) ++s;
    return s;
}

ppsp_status check_options(const ppsp_graph* g, const ppsp_options& o) {
    if (o.mode < PPSP_BIDS || o.mode > PPSP_ASTAR) return PPSP_ERR_INVALID_ARG;
    if (o.dist_bits != 32 && o.dist_bits != 64) return PPSP_ERR_INVALID_ARG;
    if (o.block_threads != 0 && o.block_threads != 256 && o.block_threads != 512 && o.block_threads != 1024)
        return PPSP_ERR_INVALID_ARG;
    if (o.frontier < PPSP_FRONTIER_AUTO || o.frontier > PPSP_FRONTIER_DENSE) return PPSP_ERR_INVALID_ARG;
    if (o.layout < PPSP_LAYOUT_AUTO || o.layout > PPSP_LAYOUT_STACKED) return PPSP_ERR_INVALID_ARG;
    if (o.batch_strategy < PPSP_BATCH_MULTI || o.batch_strategy > PPSP_BATCH_AUTO) return PPSP_ERR_INVALID_ARG;
    if ((o.batch_strategy == PPSP_BATCH_SSSP || o.batch_strategy == PPSP_BATCH_VC) && o.want_paths)
        return PPSP_ERR_UNSUPPORTED;
    if (o.team_ctas < 0 || o.big_team_ctas < 0 || o.max_ctas < 0) return PPSP_ERR_INVALID_ARG;
    if (o.ring_entries > 256) return PPSP_ERR_INVALID_ARG;
    const bool astar = o.mode == PPSP_BIDASTAR || o.mode == PPSP_ASTAR;
    if (astar && !g->info.has_coords) return PPSP_ERR_NO_COORDS;
    const bool bidir = o.mode == PPSP_BIDS || o.mode == PPSP_BIDASTAR;
    return PPSP_OK;
}

}  // namespace

static void plan_free_partial(ppsp_plan* P) {
    // a new slot may still be initialising on the plan's stream
    cudaStreamSynchronize(P->stream);
    for (Slot* x : P->slots) slot_release(P->g, x);
    P->slots.clear();
    // stream-ordered frees: no device-wide synchronisation, so plans on other
    // streams keep running (the serving loop closes plans while others run)
    if (P->d_arena && !P->host_call) cudaFreeAsync(P->d_arena, P->stream);
    if (P->d_paths) cudaFreeAsync(P->d_paths, P->stream);
    P->d_arena = nullptr;
    P->d_paths = nullptr;
    cudaGetLastError();
}

// Build everything from host pairs.  Separated so ppsp_query can reuse it.
static ppsp_status plan_create_impl(ppsp_graph* g, const uint32_t* pairs, uint64_t k, const ppsp_options* opt_in,
                                    bool single_query, ppsp_plan** out, const u64* path_caps = nullptr,
                                    bool host_call = false) {
    ppsp_options o;
    if (opt_in)
        o = *opt_in;
    else
        ppsp_options_init(&o);
    ppsp_status st = check_options(g, o);
    if (st != PPSP_OK) return st;
    if (k && !pairs) return PPSP_ERR_INVALID_ARG;
    if (o.want_paths && (!path_caps || g->info.has_zero_weight)) return PPSP_ERR_UNSUPPORTED;
    const u64 n = g->n;
    for (u64 q = 0; q < 2 * k; ++q)
        if (pairs[q] >= n) return PPSP_ERR_INVALID_ARG;
    // the graph's device order (caller ids in, device ids from here on)
    std::vector<u32> pairs_dev;
    if (!g->perm.empty()) {
        pairs_dev.resize(2 * k);
        for (u64 q = 0; q < 2 * k; ++q) pairs_dev[q] = g->perm[pairs[q]];
        pairs = pairs_dev.data();
    }

    auto P = std::make_unique<ppsp_plan>();
    P->g = g;
    P->opt = o;
    P->k = k;
    P->stream = (cudaStream_t)o.stream;
    P->dist_bits = o.dist_bits;
    const bool bidir = o.mode == PPSP_BIDS || o.mode == PPSP_BIDASTAR;
    P->memo = o.memo_potential && g->info.has_coords && (o.mode == PPSP_BIDASTAR || o.mode == PPSP_ASTAR);
    const u64 delta = o.delta ? o.delta : std::max<u64>(1, (u64)std::llround(g->info.w_mean));
    const int strategy = single_query ? PPSP_BATCH_PLAIN : o.batch_strategy;

    // ---- unique query edges ----
    P->map.assign(k, NONE);
    std::unordered_map<u64, u32> qe_id;
    std::vector<std::pair<u32, u32>> uq;  // unique queries (s, t)
    for (u64 q = 0; q < k; ++q) {
        u32 s = pairs[2 * q], t = pairs[2 * q + 1];
        if (s == t) continue;  // d(s, s) = 0, no search
        // Plain-SSSP searches from every query's own source (ordered pairs)
        const bool unordered = g->info.undirected && ((bidir && strategy != PPSP_BATCH_SSSP) ||
                                                      strategy == PPSP_BATCH_VC || strategy == PPSP_BATCH_AUTO);
        u64 key = unordered ? (((u64)std::min(s, t) << 32) | std::max(s, t)) : (((u64)s << 32) | t);
        auto it = qe_id.find(key);
        if (it == qe_id.end()) {
            it = qe_id.emplace(key, (u32)uq.size()).first;
            uq.emplace_back(s, t);
        }
        P->map[q] = it->second;  // provisional: unique-query index, renumbered below
    }
    const u32 U = (u32)uq.size();

    // ---- groups ----
    // Each group: list of vertices (searches) and list of unique-query indices.
    std::vector<std::vector<u32>> gverts, gqueries;
    std::vector<char> gsssp;                // group is one SSSP-based search (Sec. 4.3)
    // directed graphs: a query's source searches out-edges (direction 0), its
    // target in-edges (direction 1); on undirected graphs every search is 0
    const bool directed = !g->info.undirected;
    std::vector<std::vector<unsigned char>> gdirs;
    std::vector<SrcDir> sssp_src(U, SrcDir{NONE, 0});  // SSSP groups: the search answering each query
    // one SSSP group per distinct source of the queries in `qs`
    auto add_sssp_groups = [&](const std::vector<u32>& qs) {
        std::unordered_map<u64, u32> gid;
        for (u32 u : qs) {
            const u64 key = ((u64)sssp_src[u].v << 1) | sssp_src[u].dir;
            auto it = gid.find(key);
            if (it == gid.end()) {
                it = gid.emplace(key, (u32)gverts.size()).first;
                gverts.push_back({sssp_src[u].v});
                gdirs.push_back({(unsigned char)sssp_src[u].dir});
                gqueries.push_back({});
                gsssp.push_back(1);
            }
            gqueries[it->second].push_back(u);
        }
    };
    auto add_single = [&](u32 u) {
        if (bidir) {
            gverts.push_back({uq[u].first, uq[u].second});
            gdirs.push_back({0, (unsigned char)(directed ? 1 : 0)});
        } else {
            gverts.push_back({uq[u].first});
            gdirs.push_back({0});
        }
        gqueries.push_back({u});
        gsssp.push_back(0);
    };
    if (strategy == PPSP_BATCH_SSSP || strategy == PPSP_BATCH_VC) {
        // Sec. 4.3: one single-source search per selected source
        sssp_src = sssp_sources(strategy, directed, uq);
        std::vector<u32> all(U);
        std::iota(all.begin(), all.end(), 0u);
        add_sssp_groups(all);
    } else if (strategy == PPSP_BATCH_AUTO && !bidir) {
        // one search per target, except sources with several targets, which
        // get one search that stops when all of them are settled
        std::unordered_map<u32, u32> per_src;
        for (u32 u = 0; u < U; ++u) ++per_src[uq[u].first];
        std::vector<u32> multi_t;
        for (u32 u = 0; u < U; ++u) {
            if (per_src[uq[u].first] >= AUTO_MIN_TARGETS && !o.want_paths) {
                sssp_src[u] = {uq[u].first, 0};
                multi_t.push_back(u);
            } else {
                add_single(u);
            }
        }
        add_sssp_groups(multi_t);
    } else if (!bidir || (strategy != PPSP_BATCH_MULTI && strategy != PPSP_BATCH_AUTO)) {
        for (u32 u = 0; u < U; ++u) add_single(u);
    } else {
        // Multi-BiDS: V_q = distinct endpoints, components of G_q (Sec. 4.2).
        // On a directed graph V_q holds (vertex, role) pairs: a source searches
        // forward, a target backward, so G_q is bipartite (Sec. 4.4).
        std::unordered_map<u64, u32> vid;
        std::vector<u32> verts;
        std::vector<unsigned char> vrole;
        auto get = [&](u32 v, unsigned char role) {
            const u64 key = directed ? (((u64)v << 1) | role) : (u64)v;
            auto it = vid.find(key);
            if (it != vid.end()) return it->second;
            vid.emplace(key, (u32)verts.size());
            verts.push_back(v);
            vrole.push_back(directed ? role : 0);
            return (u32)verts.size() - 1;
        };
        std::vector<std::pair<u32, u32>> le(U);
        for (u32 u = 0; u < U; ++u) le[u] = {get(uq[u].first, 0), get(uq[u].second, 1)};
        UF uf((u32)verts.size());
        for (auto& e : le) uf.join(e.first, e.second);
        std::unordered_map<u32, std::vector<u32>> comp_edges;
        std::vector<u32> comp_order;
        for (u32 u = 0; u < U; ++u) {
            u32 r = uf.find(le[u].first);
            auto it = comp_edges.find(r);
            if (it == comp_edges.end()) {
                comp_order.push_back(r);
                it = comp_edges.emplace(r, std::vector<u32>()).first;
            }
            it->second.push_back(u);
        }
        const bool pot_pairs = o.mode == PPSP_BIDASTAR && g->info.has_coords;
        const bool dense = g->info.m >= AUTO_DENSE_DEG * (double)g->info.n;
        for (u32 r : comp_order) {
            const std::vector<u32>& ce = comp_edges[r];
            if (strategy == PPSP_BATCH_AUTO && (ce.size() > 1 || (dense && !pot_pairs && !o.want_paths))) {
                // the cheaper of Multi-BiDS, VC-SSSP and Plain* for this component
                std::unordered_map<u32, u32> cl;
                std::vector<std::pair<u32, u32>> cle;
                for (u32 u : ce) {
                    const u32 a = cl.emplace(le[u].first, (u32)cl.size()).first->second;
                    const u32 b = cl.emplace(le[u].second, (u32)cl.size()).first->second;
                    cle.emplace_back(a, b);
                }
                const std::vector<char> in = vertex_cover((u32)cl.size(), cle);
                u32 cover = 0;
                for (char x : in) cover += x ? 1u : 0u;
                int pick = auto_component(pot_pairs, dense, (u32)cl.size(), (u32)ce.size(), cover);
                if (pick == PPSP_BATCH_VC && o.want_paths)  // SSSP groups record no paths
                    pick = pot_pairs ? PPSP_BATCH_PLAIN_STAR : PPSP_BATCH_MULTI;
                if (pick == PPSP_BATCH_VC) {
                    // on a directed graph the component is bipartite ((vertex,
                    // role) pairs): a target in the cover searches backward
                    for (u32 j = 0; j < ce.size(); ++j)
                        sssp_src[ce[j]] = in[cle[j].first] ? SrcDir{uq[ce[j]].first, 0}
                                                           : SrcDir{uq[ce[j]].second, directed ? 1u : 0u};
                    add_sssp_groups(ce);
                    continue;
                }
                if (pick == PPSP_BATCH_PLAIN_STAR) {
                    for (u32 u : ce) add_single(u);
                    continue;
                }
            }
            // split components with more than KMAX vertices into sub-groups
            std::vector<u32> cur_v, cur_q;
            std::vector<unsigned char> cur_d;
            std::unordered_map<u32, u32> in_cur;
            for (u32 u : comp_edges[r]) {
                u32 a = le[u].first, b = le[u].second;
                u32 need = (in_cur.count(a) ? 0 : 1) + (in_cur.count(b) ? 0 : 1);
                if (cur_v.size() + need > (size_t)KMAX) {
                    gverts.push_back(cur_v);
                    gdirs.push_back(cur_d);
                    gqueries.push_back(cur_q);
                    gsssp.push_back(0);
                    cur_v.clear();
                    cur_d.clear();
                    cur_q.clear();
                    in_cur.clear();
                }
                for (u32 x : {a, b})
                    if (!in_cur.count(x)) {
                        in_cur.emplace(x, (u32)cur_v.size());
                        cur_v.push_back(verts[x]);
                        cur_d.push_back(vrole[x]);
                    }
                cur_q.push_back(u);
            }
            gverts.push_back(cur_v);
            gdirs.push_back(cur_d);
            gqueries.push_back(cur_q);
            gsssp.push_back(0);
        }
    }

    // ---- descriptors ----
    const u32 NG = (u32)gverts.size();
    std::vector<u32> uq_to_qe(U, NONE);
    std::vector<double> gwork(NG, 1.0), gdist(NG, 0.0);  // estimated work; largest heuristic distance in mean weights
    for (u32 gi = 0; gi < NG; ++gi) {
        GroupDev G{};
        const auto& V = gverts[gi];
        const auto& Q = gqueries[gi];
        G.sbeg = (u32)P->searches.size();
        G.scnt = (u32)V.size();
        G.qbeg = (u32)P->qedges.size();
        G.qcnt = (u32)Q.size();
        G.delta = delta;
        const bool sssp = gsssp[gi] != 0;
        if (sssp) {
            G.mode = GM_SSSP;
            G.target = NONE;
        } else if (bidir) {
            G.mode = GM_BIDIR;
            G.target = NONE;
        } else {
            G.mode = (o.mode == PPSP_ASTAR) ? GM_ASTAR : GM_ET;
            G.target = uq[Q[0]].second;
        }
        if (G.scnt <= 2) {
            G.layout = PPSP_LAYOUT_INTERLEAVED;
            G.kshift = (G.scnt == 2) ? 1 : 0;
        } else {
            G.layout = (o.layout == PPSP_LAYOUT_STACKED) ? PPSP_LAYOUT_STACKED : PPSP_LAYOUT_INTERLEAVED;
            G.kshift = ceil_log2(G.scnt);
        }
        const u64 range = G.layout == PPSP_LAYOUT_INTERLEAVED ? (n << G.kshift) : (u64)G.scnt * n;
        if (range >= 0xFFFFFFFFull) return PPSP_ERR_UNSUPPORTED;
        const auto& Dv = gdirs[gi];
        std::unordered_map<u64, u32> local;  // (vertex, direction) -> search
        auto lkey = [](u32 v, unsigned char d) { return ((u64)v << 1) | d; };
        for (u32 i = 0; i < G.scnt; ++i) local.emplace(lkey(V[i], Dv[i]), i);
        const unsigned char tdir = directed ? 1 : 0;  // direction of a query's target search
        std::vector<std::vector<PartnerDev>> plist(G.scnt);
        std::vector<i64> hmax(G.scnt, 0);
        double work = 0.0;
        for (u32 qi = 0; qi < G.qcnt; ++qi) {
            u32 u = Q[qi];
            u32 qe = G.qbeg + qi;
            uq_to_qe[u] = qe;
            QEdgeDev e;
            if (sssp) {
                // one search; b holds the query's other endpoint (a vertex id)
                e.a = 0;
                e.b = (uq[u].first == sssp_src[u].v && sssp_src[u].dir == 0) ? uq[u].second : uq[u].first;
            } else {
                e.a = local[lkey(uq[u].first, 0)];
                e.b = bidir ? local[lkey(uq[u].second, tdir)] : e.a;
            }
            P->qedges.push_back(e);
            P->qedge_ends.emplace_back(uq[u].first, uq[u].second);
            if (bidir && !sssp) {
                plist[e.a].push_back(PartnerDev{e.b, qe});
                plist[e.b].push_back(PartnerDev{e.a, qe});
            }
            i64 h = g->info.has_coords ? pot_h_host(g, uq[u].first, uq[u].second) : 1;
            hmax[e.a] = std::max(hmax[e.a], h);
            if (!sssp) hmax[e.b] = std::max(hmax[e.b], h);
        }
        for (u32 i = 0; i < G.scnt; ++i) {
            SearchDev s{};
            s.src = V[i];
            s.dir = Dv[i];
            s.pbeg = (u32)P->partners.size();
            s.pcnt = (u32)plist[i].size();
            for (auto& pd : plist[i]) P->partners.push_back(pd);
            s.pot = 0;
            s.pot_b = V[i];
            s.key_off = 0;
            if (sssp) {
                // no pruning, no potential
            } else if (o.mode == PPSP_BIDASTAR && G.scnt == 2) {
                // Sec. 3.5 for an isolated pair: rho_i = h_partner - h_self, so the
                // two searches use exactly opposite potentials (h_F = -h_B, which
                // Theorem 3.4 relies on).
                s.pot = 1;
                s.pot_b = V[plist[i][0].j];
                s.key_off = -pot_h_host(g, s.pot_b, s.src);
            } else if (o.mode == PPSP_BIDASTAR && o.multi_potential && g->info.has_coords && !plist[i].empty()) {
                // a shared search cannot hold the opposite of every partner's
                // potential at once.  By default it runs without one (plain
                // Multi-BiDS); with multi_potential it takes the smallest
                // partner potential (multi-target A*), so that for every query
                // (i, j) it prunes no more than the pair's BiD-A* rule would;
                // the key is shifted so that the source's key is 0
                s.pot = 2;
                i64 hmin = INT64_MAX;
                for (const PartnerDev& pd : plist[i]) hmin = std::min(hmin, pot_h_host(g, V[pd.j], s.src));
                s.key_off = -hmin;
            } else if (o.mode == PPSP_ASTAR && !sssp) {
                s.pot_b = G.target;
                s.key_off = -pot_h_host(g, G.target, s.src);
            }
            P->searches.push_back(s);
            // estimated settled area: a disc of radius hmax / 2 per search of a
            // pruned bidirectional group, of radius hmax for an SSSP group
            work += (double)(hmax[i] + 1) * (double)(hmax[i] + 1) / (sssp ? 1.0 : 4.0);
        }
        gwork[gi] = work;
        gdist[gi] = (double)*std::max_element(hmax.begin(), hmax.end()) / std::max(1e-9, g->info.w_mean);
        if (o.delta == 0 && g->delta_model[o.mode] == nullptr && g->growth == GROWTH_PLANE &&
            (G.mode == GM_ASTAR || (G.mode == GM_BIDIR && P->searches[G.sbeg].pot == 1)))
            G.delta = std::max<u64>(1, (u64)std::llround((double)delta / astar_divisor(bidir, gdist[gi])));
        P->groups.push_back(G);
    }
    for (u64 q = 0; q < k; ++q)
        if (P->map[q] != NONE) P->map[q] = uq_to_qe[P->map[q]];

    // ---- features of the learned stepping increment (per group) ----
    // raw: heuristic distance, deg(s), deg(t), w mean/std/min/max, n, m,
    // |V_q|, |E_q|, mean query-graph degree; the model sees log2(1 + raw).
    P->delta_default = delta;
    P->feats.assign((size_t)NG * 12, 0.f);
    for (u32 gi = 0; gi < NG; ++gi) {
        const GroupDev& G = P->groups[gi];
        double hsum = 0.0;
        for (u32 qi = 0; qi < G.qcnt; ++qi) {
            auto ends = P->qedge_ends[G.qbeg + qi];
            if (g->info.has_coords) hsum += (double)pot_h_host(g, ends.first, ends.second);
        }
        double dmean = 0.0, dmax = 0.0;
        for (u32 i = 0; i < G.scnt; ++i) {
            double d = (double)g->deg[P->searches[G.sbeg + i].src];
            dmean += d / G.scnt;
            dmax = std::max(dmax, d);
        }
        double ds = (double)g->deg[P->searches[G.sbeg].src];
        double dt = G.scnt >= 2 ? (double)g->deg[P->searches[G.sbeg + 1].src]
                                : (G.target != NONE ? (double)g->deg[G.target] : 0.0);
        if (G.scnt > 2) {
            ds = dmean;
            dt = dmax;
        }
        const double raw[12] = {hsum / std::max<u32>(1, G.qcnt), ds, dt, g->info.w_mean, g->info.w_std,
                                (double)g->info.w_min, (double)g->info.w_max, (double)g->n, (double)g->m,
                                (double)G.scnt, (double)G.qcnt, 2.0 * G.qcnt / std::max<u32>(1, G.scnt)};
        for (int f = 0; f < 12; ++f) P->feats[(size_t)gi * 12 + f] = (float)std::log2(1.0 + std::max(0.0, raw[f]));
    }
    // the models were trained on pair and Multi-BiDS groups: the inference
    // kernel leaves SSSP groups at the default increment
    if (o.delta == 0 && g->delta_model[o.mode] != nullptr) P->model = g->delta_model[o.mode];

    // ---- launch shape ----
    // teams of several CTAs: 512 threads (128 registers), or 1,024 (64) where
    // rows are long and the edge loop, which needs few registers, dominates
    // (RMAT-20: 75 groups 174 against 130 ms on teams of eight).  Not on
    // graphs with long rows that grow as in the plane (nearest-neighbour
    // graphs), whose steps are short (2^18 vertices, eight neighbours each: 8
    // BiDS queries one at a time 13.8 against 11.1 ms, 24 pairs 4.8 on 1,024
    // threads and teams of eight against 4.0)
    const bool hubs = g->wsorted && g->growth != GROWTH_PLANE;
    int block = o.block_threads ? o.block_threads : (hubs ? 1024 : 512);
    int bpsm = 0, sms = 0;
    u32 ring_cap = o.ring_entries ? o.ring_entries : RING_CAP_DEFAULT;
    st = engine_occupancy(o.dist_bits, block, &bpsm, &sms, ENGINE_GENERAL, ring_cap);
    if (st != PPSP_OK) return st;
    if (bpsm < 1) return PPSP_ERR_UNSUPPORTED;
    u32 grid = (u32)(bpsm * sms);
    if (o.max_ctas > 0) grid = std::min<u32>(grid, (u32)o.max_ctas);
    P->block = block;

    // ---- teams and queues ----
    std::vector<u32> big, small;
    bool any_sssp = false;
    for (u32 gi = 0; gi < NG; ++gi) {
        (P->groups[gi].scnt > 2 ? big : small).push_back(gi);
        any_sssp = any_sssp || P->groups[gi].mode == GM_SSSP;
    }
    auto by_work = [&](u32 a, u32 b) { return gwork[a] > gwork[b]; };
    std::stable_sort(big.begin(), big.end(), by_work);
    std::stable_sort(small.begin(), small.end(), by_work);
    struct TeamSpec {
        u32 size, queue;
    };
    // Small graphs with long rows: a team's step on the queue path is a chain of
    // barriers and atomics that are waited for, 17 to 50 us whatever the team's
    // size, so one CTA with its buckets in shared memory is faster while a step
    // fits it.  RMAT-11 / 13 / 15 / 16, ten BiDS queries one at a time: 4.9,
    // 8.0, 9.1, 30.7 ms on all CTAs, 2.4, 4.0, 7.6, 29.7 on one; 24 pairs at
    // once 0.75, 2.2, 3.6, 4.3 against 0.37, 0.95, 2.1, 3.6.  Single-source
    // groups scan more: 90 of them 1.5, 4.7, 16.4, 24.9 against 0.57, 2.4, 14.1,
    // 31.0, but 24 of them 0.6, 1.5, 6.2, 8.9 against 0.5, 2.0, 9.7, 26.
    const bool small_dense = g->wsorted && !any_sssp && g->m <= (1u << 20);
    const bool small_sssp = g->wsorted && any_sssp && g->m <= (1u << 19);
    // teams for `grid` resident CTAs; returns the CTAs they use
    auto build_teams = [&](u32 grid_in, std::vector<TeamSpec>& teams) -> u32 {
        teams.clear();
        u32 g_used = grid_in;
        if (strategy == PPSP_BATCH_PLAIN) {
            // one query (group) at a time on the whole GPU
            u32 ts = o.team_ctas ? std::min<u32>(grid_in, (u32)o.team_ctas) : small_dense ? 1u : grid_in;
            g_used = ts;
            teams.push_back({ts, 1});
            P->queue_items[0].clear();
            P->queue_items[1] = big;
            P->queue_items[1].insert(P->queue_items[1].end(), small.begin(), small.end());
        } else {
            double wb = 0, ws = 0;
            for (u32 gi : big) wb += gwork[gi];
            for (u32 gi : small) ws += gwork[gi];
            u32 g_big = 0;
            if (!big.empty() && small.empty())
                g_big = grid_in;
            else if (!big.empty())
                g_big = std::min<u32>(grid_in - 1, std::max<u32>(1, (u32)std::llround(grid_in * wb / (wb + ws))));
            u32 tb = 0, nbt = 0;
            if (g_big) {
                nbt = std::min<u32>((u32)big.size(), g_big);
                tb = o.big_team_ctas ? std::min<u32>((u32)o.big_team_ctas, g_big) : g_big / nbt;
                nbt = std::max<u32>(1, std::min<u32>(g_big / tb, (u32)big.size()));
                for (u32 t = 0; t < nbt; ++t) teams.push_back({tb, 0});
            }
            u32 g_small = grid_in - nbt * tb;
            if (!small.empty() && g_small > 0) {
                // fewer groups than CTAs: give each group a team of several CTAs
                u32 ts_auto = 1;
                while (ts_auto * 2 <= 32 && (u64)ts_auto * 2 * small.size() <= g_small) ts_auto *= 2;
                // Graphs with long rows and hubs (RMAT shapes): eight CTAs at least,
                // which take the groups in turn, longest first: a group's
                // steps are large enough to share, and the longest one (a
                // search with many targets) no longer outlasts the rest.
                // RMAT-20, teams of 2 / 4 / 8 / 16: 75 single-source groups
                // 225 / 160 / 130 / 195 ms, 24 of them 172 / 88 / 51 / 56, 300
                // 468 / 377 / 375 / 576 (one CTA each: 2,490), 24 pairs 199 /
                // 98 / 54 / 34.  More pairs than CTAs stay on one CTA each
                // (300: 205 against 231).
                if (small_dense || (small_sssp && small.size() * 4 > g_small))
                    ts_auto = 1;
                else if (hubs && (any_sssp || small.size() <= g_small))
                    ts_auto = std::max<u32>(ts_auto, std::min<u32>(8, g_small));
                u32 ts = o.team_ctas ? std::min<u32>((u32)o.team_ctas, g_small) : ts_auto;
                // no more teams than groups: an idle team would still hold a slot
                u32 nst = std::max<u32>(1, std::min<u32>(g_small / ts, (u32)small.size()));
                for (u32 t = 0; t < nst; ++t) teams.push_back({ts, 1});
                g_small = nst * ts;
            } else {
                g_small = 0;
            }
            g_used = nbt * tb + g_small;
            P->queue_items[0] = big;
            P->queue_items[1] = small;
        }
        if (teams.empty() || g_used == 0) {
            teams.assign(1, {1, 1});
            g_used = 1;
        }
        return g_used;
    };
    auto all_single = [](const std::vector<TeamSpec>& teams) {
        bool one = !teams.empty();
        for (auto& tm : teams) one = one && tm.size == 1;
        return one;
    };
    std::vector<TeamSpec> teams;
    const u32 grid_max = grid;  // resident CTAs of the general kernel

    // ---- kernel ----
    // On a graph with adjacency blocks, groups of one or two searches run the
    // bucketed kernel, one CTA each, however few they are (the step of such a
    // group has a few hundred entries, which one CTA takes in less time than
    // several need to meet at a barrier), and larger groups run one CTA per
    // search.  What that kernel does not do stays with the others: explicit
    // team sizes, a forced frontier or layout, merged buckets (rho), memoized
    // potentials, the pull step, multi-target potentials, paths of larger
    // groups and the barrier test hook.
    const bool plain_opts = o.frontier == PPSP_FRONTIER_AUTO && o.debug_flags == 0;
    bool bucket = plain_opts && g->d_blk8 && o.team_ctas <= 1 && !o.stepping_rho && !P->memo &&
                  !(o.pull_push && g->info.undirected);
    u32 tsize = 0;  // CTAs of a team for the larger groups: the most searches of one
    for (u32 gi : big) {
        tsize = std::max(tsize, P->groups[gi].scnt);
        bucket = bucket && P->groups[gi].layout == PPSP_LAYOUT_INTERLEAVED;
    }
    if (tsize && (o.big_team_ctas || o.multi_potential || o.want_paths || strategy == PPSP_BATCH_PLAIN)) bucket = false;
    if (bucket) {
        bool all_bidir = true;
        for (const GroupDev& G : P->groups) all_bidir = all_bidir && G.mode == GM_BIDIR;
        const bool plain = strategy == PPSP_BATCH_PLAIN;
        const u64 ctas = plain ? std::max<u32>(1, tsize) : small.size() + (u64)tsize * big.size();
        const bool one = !plain && (o.team_ctas == 1 || 2 * P->groups.size() > grid_max);
        bucket = blocks_pay(g, all_bidir, one, tsize == 0, ctas, (u32)sms);
    }
    // CTAs of 256 threads take four times as long for a step of a few hundred
    // entries, and no cluster of them is compiled: few searches without a
    // potential share the queue path (BiDS, 24 pairs on a 700^2 road graph 34.5 ms
    // on one CTA each, 9.4 there; BiD-A* 8.2 against 23).
    if (bucket && o.block_threads == 256 && !o.team_ctas && !tsize &&
        (strategy == PPSP_BATCH_PLAIN || 2 * P->groups.size() <= grid_max))
        for (u32 gi : small) bucket = bucket && (P->groups[gi].mode == GM_ASTAR || P->searches[P->groups[gi].sbeg].pot != 0);
    // An explicit increment far above the best one makes few steps of many
    // thousand entries, which a large team shares better: few groups with one
    // go to the queue path, as all did before.  One BiD-A* query at a time on
    // the 2048^2 road graph with one mean weight: 1,950 ms on one CTA or a
    // cluster, 44 to 66 on teams of 16, 12 to 16 on all CTAs.
    if (bucket && o.delta && !o.team_ctas && (strategy == PPSP_BATCH_PLAIN || 2 * P->groups.size() <= grid_max)) {
        double div = 0.5;
        for (u32 gi : small)
            if (P->searches[P->groups[gi].sbeg].pot)
                div = std::max(div, astar_divisor(P->groups[gi].mode == GM_BIDIR, gdist[gi]) / 1.5);
        if ((double)o.delta * div > g->info.w_mean) bucket = false;
    }
    // Whether `count` slots are idle in the graph's pool or fit half of the
    // memory that is free now.
    auto slots_free = [&](const SlotCaps& sc, u64 count) {
        u64 idle = 0;
        for (auto it = g->idle.lower_bound(SlotKey{o.dist_bits, sc.flat_cap, 0, 0, false});
             it != g->idle.end() && it->first.dist_bits == o.dist_bits && it->first.flat_cap <= 2 * sc.flat_cap + 4096; ++it)
            idle += it->first.qcap >= sc.qcap && it->first.tcap >= sc.tcap;
        if (idle >= count) return true;
        size_t free_b = 0, total_b = 0;
        if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
            cudaGetLastError();
            return true;
        }
        return (count - idle) * slot_alloc_bytes(o.dist_bits, sc.flat_cap, sc.qcap, sc.tcap) <= free_b / 2;
    };
    if (bucket) {
        EngineKind kind = tsize ? ENGINE_BUCKET_TEAMS : ENGINE_BUCKET;
        const u64 want = small.size() + (u64)tsize * big.size();  // CTAs that run everything at once
        u64 small_range = 0;
        for (u32 gi : small) small_range = std::max<u64>(small_range, n << P->groups[gi].kshift);
        int bb = o.block_threads;
        if (!bb) {
            // Two groups per SM (512 threads each) when enough of them run at
            // once to fill both (not one at a time, nor on max_ctas CTAs that
            // fit the SMs) and the slots of twice the teams leave most of
            // the memory free; otherwise one group of 1,024 threads, which
            // finishes sooner.  Measured: 1,000 queries on the 1024^2 road
            // graph 16.4 against 17.6 ms, 2,048 on the 2048^2 one 100 against
            // 115 ms; 256 queries on the 4096^2 one 247 against 136 ms.
            const SlotCaps sc = slot_caps(small_range, o.frontier, false);
            const u64 two = 2ull * sms * slot_alloc_bytes(o.dist_bits, sc.flat_cap, sc.qcap, sc.tcap);
            const bool both = strategy != PPSP_BATCH_PLAIN && want > 4 * (u64)sms &&
                              (!o.max_ctas || 2 * (u64)o.max_ctas > 3 * (u64)sms);
            bb = (both && two <= g->device_mem / 4 && slots_free(sc, 2ull * sms)) ? 512 : 1024;
        }
        const u32 cap = bucket_cap(o.ring_entries, bb, o.dist_bits);
        const u32 long_cap = bucket_cap(o.ring_entries, 1024, o.dist_bits);
        // A cluster of CTAs per group where there are too few groups for the
        // SMs and their steps are large, or the longest groups would outlast
        // the rest: the smallest estimated time, by a tenth at least.
        auto group_us = [&](u32 gi, u32 k, double busy = 0.0, int threads = 1024) {
            const GroupDev& G = P->groups[gi];
            // without a potential on a scale (no coordinates, or none that the
            // weights allow) the length of a query of a square grid
            const bool scaled = g->info.has_coords && g->pot_scale > 0.0;
            const double H = scaled ? gdist[gi] : std::sqrt((double)n) / 2;
            const u32 mode = !scaled && G.mode == GM_ASTAR ? (u32)GM_ET : G.mode;
            return bucket_group_us(mode, scaled && P->searches[G.sbeg].pot != 0, H, (double)n, k, busy, threads);
        };
        u32 cl = 1, ncl = 0;
        double alone = 0;  // estimated time of the groups in one launch
        bool all_pairs_pot = !tsize;  // BiD-A* pairs only
        for (u32 gi : small)
            all_pairs_pot = all_pairs_pot && P->groups[gi].mode == GM_BIDIR && P->searches[P->groups[gi].sbeg].pot && g->pot_scale > 0.0;
        if (!tsize && !o.want_paths && !o.team_ctas && bb >= 512 &&
            (bb == 1024 || o.block_threads) && !small.empty()) {
            double best = 0;
            for (u32 k = 1; k <= 8; k *= 2) {
                int nteams = sms;
                if (k > 1) {
                    st = engine_clusters(o.dist_bits, bb, cap, k, &nteams);
                    if (st != PPSP_OK) return st;
                }
                if (o.max_ctas > 0) nteams = std::min<int>(nteams, o.max_ctas / (int)k);
                if (strategy == PPSP_BATCH_PLAIN) nteams = std::min(nteams, 1);
                if (nteams < 1) break;
                double sum = 0, most = 0;
                for (u32 gi : small) {
                    const double us = group_us(gi, k, all_pairs_pot && small.size() * k > (size_t)sms ? CLUSTER_BUSY : 0.0, bb);
                    sum += us;
                    most = std::max(most, us);
                }
                const double us = std::max(sum / std::min<double>(nteams, (double)small.size()), most);
                if (k == 1 || us < 0.9 * best) {
                    best = us;
                    cl = k;
                    ncl = (u32)nteams;
                }
            }
            if (cl > 1) kind = ENGINE_BUCKET_CLUSTERS;
            alone = best;
        }
        // The longest groups on more threads each, beside the rest.
        LongGroups lg;
        if (all_pairs_pot && (bb == 1024 || !o.block_threads) && !o.max_ctas && !o.team_ctas &&
            strategy != PPSP_BATCH_PLAIN && small.size() > 1) {
            const u32 per_sm = bb == 512 ? 2 : 1;
            std::vector<double> us[4];
            u32 most[4] = {(u32)sms, 0, 0, 0};
            for (u32 c = 0; c < (o.want_paths ? 1u : 4u); ++c) {
                int nt = sms;
                if (c) {
                    st = engine_clusters(o.dist_bits, 1024, long_cap, 1u << c, &nt);
                    if (st != PPSP_OK) return st;
                }
                most[c] = (u32)std::max(nt, 0);
                for (u32 gi : small) us[c].push_back(group_us(gi, 1u << c, CLUSTER_BUSY));
            }
            if (bb == 512) {
                double sum = 0, longest = 0;
                for (double x : us[0]) {
                    sum += x;
                    longest = std::max(longest, x);
                }
                alone = std::max(LONG_512 * LONG_SPREAD * longest, GROUP_512 * sum / std::min<double>(2.0 * sms, (double)small.size()));
            }
            if (alone > 0) lg = long_groups(us, most, (u32)sms, per_sm, alone);
            const SlotCaps sc = slot_caps(small_range, o.frontier, false);
            const u64 slots = lg.teams + std::min<u64>(small.size() - lg.groups, (u64)per_sm * sms);
            if (lg.groups && (slots * slot_alloc_bytes(o.dist_bits, sc.flat_cap, sc.qcap, sc.tcap) > g->device_mem / 2 ||
                              !slots_free(sc, slots)))
                lg = LongGroups();
            if (lg.groups) {
                kind = ENGINE_BUCKET;
                cl = 1;
            }
        }
        int bbpsm = 0, bsms = 0;
        st = engine_occupancy(o.dist_bits, bb, &bbpsm, &bsms, cl > 1 ? ENGINE_BUCKET : kind, cap);
        if (st != PPSP_OK) return st;
        u32 res = (u32)(bbpsm * bsms);
        if (o.max_ctas > 0) res = std::min<u32>(res, (u32)o.max_ctas);
        // teams for the larger groups: one each when everything fits, else
        // by their share of the estimated work
        u32 nbt = 0;
        if (tsize) {
            double wb = 0, ws = 0;
            for (u32 gi : big) wb += gwork[gi];
            for (u32 gi : small) ws += gwork[gi];
            const u32 room = small.empty() ? res : res - std::min<u32>(res, 1);
            nbt = want <= res ? (u32)big.size()
                              : std::min<u32>((u32)big.size(),
                                              std::max<u32>(1, std::min<u32>(room, (u32)(res * wb / (wb + ws))) / tsize));
        }
        if (bbpsm >= 1 && res >= 1 && (u64)nbt * tsize + (small.empty() ? 0 : 1) <= res) {
            const u32 left = res - nbt * tsize;
            const u32 ns = small.empty() ? (tsize ? 0u : 1u)
                                         : (strategy == PPSP_BATCH_PLAIN ? 1u : std::min<u32>(left, (u32)small.size()));
            teams.assign(nbt, {tsize, 0});
            teams.insert(teams.end(), cl > 1 ? std::min<u32>(ncl, (u32)small.size()) : ns, {cl, 1});
            if (strategy == PPSP_BATCH_PLAIN && cl > 1) teams.resize(1);
            if (lg.groups) {
                teams.assign(lg.teams, {lg.cl, 0});
                teams.insert(teams.end(), std::min<u32>(res, (u32)small.size() - lg.groups), {1, 1});
            }
            grid = 0;
            for (const TeamSpec& tm : teams) grid += tm.size;
            P->args.cluster = lg.groups ? lg.cl : cl;
            P->args.long_ctas = lg.teams * lg.cl;
            P->args.long_cap = long_cap;
            P->queue_items[0] = big;
            P->queue_items[1] = small;
            if (lg.groups) {  // no larger groups here
                P->queue_items[0].assign(small.begin(), small.begin() + lg.groups);
                P->queue_items[1].assign(small.begin() + lg.groups, small.end());
            }
            P->block = bb;
            P->kind = kind;
            ring_cap = cap;
        }
    }
    if (P->kind == ENGINE_GENERAL) grid = build_teams(grid_max, teams);

    // ---- block size ----
    // Every team of one CTA runs the bucketed shared-memory path, in the
    // kernel instance without the queue / bitmap path (fewer registers):
    // by default one CTA of 1,024 threads per SM (one group per CTA then
    // finishes sooner: on the road benchmark the longest query drops from 34
    // to 25 ms and the batch from 38.3 to 36.8 ms); block_threads = 512 or
    // 256 gives two or four CTAs per SM, each running its own group.  Teams
    // of several CTAs keep 512 threads (128 registers, no spills on the queue
    // path).  The barrier test hook needs the team barrier, so not with it.
    if (P->kind == ENGINE_GENERAL && plain_opts && all_single(teams)) {
        const int lb = o.block_threads ? o.block_threads : 1024;
        int lbpsm = 0, lsms = 0;
        if (engine_occupancy(o.dist_bits, lb, &lbpsm, &lsms, ENGINE_LOCAL, ring_cap) == PPSP_OK && lbpsm >= 1) {
            u32 lgrid = (u32)(lbpsm * lsms);
            if (o.max_ctas > 0) lgrid = std::min<u32>(lgrid, (u32)o.max_ctas);
            if (lgrid >= grid) {
                std::vector<TeamSpec> t2;
                const u32 g2 = build_teams(lgrid, t2);
                if (all_single(t2)) {
                    teams.swap(t2);
                    grid = g2;
                } else {
                    // the first layout (all single), rebuilt from the same
                    // input so that its queues are restored with it
                    grid = build_teams(grid_max, teams);
                }
                P->block = lb;
                P->kind = ENGINE_LOCAL;
            }
        }
    }
    if (o.delta == 0 && g->delta_model[o.mode] == nullptr && g->growth != GROWTH_PLANE && all_single(teams))
        for (u32 gi = 0; gi < NG; ++gi)
            if (P->groups[gi].mode == GM_ASTAR)
                P->groups[gi].delta =
                    std::max<u64>(1, (u64)std::llround((double)delta / astar_divisor(false, gdist[gi])));
    P->grid = grid;
    u32 first = 0;
    for (u32 t = 0; t < teams.size(); ++t) {
        P->team_first.push_back(first);
        P->team_size.push_back(teams[t].size);
        P->team_queue.push_back(teams[t].queue);
        for (u32 c = 0; c < teams[t].size; ++c) P->cta_team.push_back(t);
        first += teams[t].size;
    }
    // every launched CTA belongs to exactly one team (a CTA without one would
    // read past the team tables)
    if (first != grid || grid == 0) {
        set_last_internal_error("team layout covers %u CTAs of a grid of %u", first, grid);
        return PPSP_ERR_CUDA;
    }

    // ---- slots ----
    u64 range_q[MAX_QUEUES] = {0, 0};
    for (u32 qd = 0; qd < MAX_QUEUES; ++qd)
        for (u32 gi : P->queue_items[qd]) {
            const GroupDev& G = P->groups[gi];
            u64 range = G.layout == PPSP_LAYOUT_INTERLEAVED ? (n << G.kshift) : (u64)G.scnt * n;
            range_q[qd] = std::max(range_q[qd], range);
        }
    for (u32 t = 0; t < teams.size(); ++t) {
        const SlotCaps sc = slot_caps(range_q[teams[t].queue], o.frontier, teams[t].size == grid);
        Slot* s = nullptr;
        st = slot_acquire(g, o.dist_bits, sc.flat_cap, sc.qcap, sc.tcap, P->memo, P->stream, &s);
        if (st == PPSP_ERR_OOM && P->kind >= ENGINE_BUCKET && teams[t].queue == 1 && t > 0 && teams[t - 1].queue == 1) {
            // the teams of a queue take its groups in turn: run with fewer
            grid = P->team_first[t];
            P->grid = grid;
            P->cta_team.resize(grid);
            P->team_first.resize(t);
            P->team_size.resize(t);
            P->team_queue.resize(t);
            teams.resize(t);
            break;
        }
        if (st != PPSP_OK) {
            cudaStreamSynchronize(P->stream);  // new slots may still be initialising
            cudaGetLastError();
            for (Slot* x : P->slots) slot_release(g, x);
            return st;
        }
        P->slots.push_back(s);
    }

    // ---- device arena ----
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const u32 NT = (u32)teams.size();
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o2 = off;
        off += al(std::max<size_t>(bytes, 1));
        return o2;
    };
    size_t o_groups = take(P->groups.size() * sizeof(GroupDev));
    size_t o_search = take(P->searches.size() * sizeof(SearchDev));
    size_t o_part = take(P->partners.size() * sizeof(PartnerDev));
    size_t o_qe = take(P->qedges.size() * sizeof(QEdgeDev));
    size_t o_ctat = take(P->cta_team.size() * 4);
    size_t o_tf = take(NT * 4), o_tsz = take(NT * 4), o_tq = take(NT * 4);
    size_t o_slots = take(NT * sizeof(SlotDev));
    size_t o_q0 = take(P->queue_items[0].size() * 4), o_q1 = take(P->queue_items[1].size() * 4);
    size_t o_map = take(k * 4);
    size_t o_feat = take(P->feats.size() * 4);
    size_t static_bytes = off;
    // run state (zero when a run starts), then what a run leaves: the error
    // word, the counters and mu lie together, so that one copy brings them back
    size_t o_run = off;
    size_t o_qh = take(MAX_QUEUES * 4);
    size_t o_ts = take(NT * sizeof(TeamState));
    size_t o_gns = take(P->groups.size() * 8);
    size_t o_err = take(4);
    size_t o_cnt = take(sizeof(EngineCounters));
    P->runstate_bytes = off - o_run;
    size_t o_mu = take(P->qedges.size() * 8);
    P->back_at = o_err;
    P->back_bytes = o_mu + P->qedges.size() * 8 - o_err;
    size_t o_mumax = take(P->searches.size() * 8);
    P->arena_bytes = off;
    const size_t up_bytes = host_call ? o_run + P->runstate_bytes : static_bytes;
    cudaError_t ce = cudaSuccess;
    if (host_call && g->ws.reserve(P->arena_bytes, std::max(up_bytes, P->back_bytes), P->stream)) {
        P->host_call = true;
        P->d_arena = g->ws.dev;
    } else if (host_call) {
        ce = cudaErrorMemoryAllocation;
    } else {
        ce = cudaMallocAsync(&P->d_arena, P->arena_bytes, P->stream);
    }
    if (ce != cudaSuccess) {
        cudaGetLastError();
        cudaStreamSynchronize(P->stream);  // new slots may still be initialising
        cudaGetLastError();
        for (Slot* x : P->slots) slot_release(g, x);
        return ce == cudaErrorMemoryAllocation ? PPSP_ERR_OOM : PPSP_ERR_CUDA;
    }
    char* base = (char*)P->d_arena;
    std::vector<char> pageable(host_call ? 0 : static_bytes, 0);
    char* h = host_call ? g->ws.host : pageable.data();
    if (host_call) memset(h, 0, up_bytes);
    auto put = [&](size_t o2, const void* src, size_t bytes) {
        if (bytes) memcpy(h + o2, src, bytes);
    };
    put(o_groups, P->groups.data(), P->groups.size() * sizeof(GroupDev));
    put(o_search, P->searches.data(), P->searches.size() * sizeof(SearchDev));
    put(o_part, P->partners.data(), P->partners.size() * sizeof(PartnerDev));
    put(o_qe, P->qedges.data(), P->qedges.size() * sizeof(QEdgeDev));
    put(o_ctat, P->cta_team.data(), P->cta_team.size() * 4);
    put(o_tf, P->team_first.data(), NT * 4);
    put(o_tsz, P->team_size.data(), NT * 4);
    put(o_tq, P->team_queue.data(), NT * 4);
    std::vector<SlotDev> sd(NT);
    for (u32 t = 0; t < NT; ++t) sd[t] = P->slots[t]->dev;
    put(o_slots, sd.data(), NT * sizeof(SlotDev));
    put(o_q0, P->queue_items[0].data(), P->queue_items[0].size() * 4);
    put(o_q1, P->queue_items[1].data(), P->queue_items[1].size() * 4);
    put(o_map, P->map.data(), k * 4);
    put(o_feat, P->feats.data(), P->feats.size() * 4);
    // a pageable source is staged before the call returns, so it may go out of
    // scope; the workspace stays until the call's work has ended
    ce = cudaMemcpyAsync(base, h, up_bytes, cudaMemcpyHostToDevice, P->stream);
    if (ce != cudaSuccess) {
        cudaGetLastError();
        plan_free_partial(P.get());
        return PPSP_ERR_CUDA;
    }

    EngineArgs& a = P->args;
    a.g = g->dev();
    a.groups = (const GroupDev*)(base + o_groups);
    a.searches = (const SearchDev*)(base + o_search);
    a.partners = (const PartnerDev*)(base + o_part);
    a.qedges = (const QEdgeDev*)(base + o_qe);
    a.mu = (u64*)(base + o_mu);
    a.mumax = (u64*)(base + o_mumax);
    a.cta_team = (const u32*)(base + o_ctat);
    a.team_first = (const u32*)(base + o_tf);
    a.team_size = (const u32*)(base + o_tsz);
    a.team_queue = (const u32*)(base + o_tq);
    a.tstate = (TeamState*)(base + o_ts);
    a.slots = (SlotDev*)(base + o_slots);
    a.queue_items[0] = (const u32*)(base + o_q0);
    a.queue_items[1] = (const u32*)(base + o_q1);
    a.queue_len[0] = (u32)P->queue_items[0].size();
    a.queue_len[1] = (u32)P->queue_items[1].size();
    a.queue_head = (u32*)(base + o_qh);
    a.dense_den = o.dense_den ? o.dense_den : 16u;
    a.frontier = (u32)o.frontier;
    a.rho = o.stepping_rho;
    a.memo = P->memo ? 1u : 0u;
    a.ring_cap = ring_cap;
    a.pull = (o.pull_push && g->info.undirected) ? 1u : 0u;
    a.split = (!a.pull && g->info.deg_max > ROW_CHUNK) ? 1u : 0u;
    a.debug = o.debug_flags;
    a.spin_limit = o.spin_limit ? o.spin_limit : (1ull << 26);
    a.err = (u32*)(base + o_err);
    a.counters = (EngineCounters*)(base + o_cnt);
    a.group_ns = (u64*)(base + o_gns);
    P->d_runstate = base + o_run;
    P->d_map = (u32*)(base + o_map);
    P->d_feats = (float*)(base + o_feat);
    if (o.want_paths) {
        const u64 NQ = P->qedges.size();
        std::vector<u64> cap(NQ, 0);
        for (u64 q = 0; q < k; ++q)
            if (P->map[q] != NONE) cap[P->map[q]] = std::max(cap[P->map[q]], path_caps[q]);
        P->path_off.assign(NQ + 1, 0);
        for (u64 e = 0; e < NQ; ++e) P->path_off[e + 1] = P->path_off[e] + cap[e];
        const size_t b_buf = ((P->path_off[NQ] * 4) + 255) & ~(size_t)255;
        const size_t b_off = ((NQ + 1) * 8 + 255) & ~(size_t)255;
        const size_t b_len = (NQ * 8 + 255) & ~(size_t)255;
        const size_t b_meet = (NQ * 4 + 255) & ~(size_t)255;
        ce = cudaMallocAsync(&P->d_paths, std::max<size_t>(256, b_buf + b_off + b_len + b_meet), P->stream);
        if (ce != cudaSuccess) {
            cudaGetLastError();
            plan_free_partial(P.get());
            return ce == cudaErrorMemoryAllocation ? PPSP_ERR_OOM : PPSP_ERR_CUDA;
        }
        char* pb = (char*)P->d_paths;
        a.path_buf = (u32*)pb;
        a.path_off = (const u64*)(pb + b_buf);
        a.path_len = (u64*)(pb + b_buf + b_off);
        P->d_meet = (u32*)(pb + b_buf + b_off + b_len);
        a.meet = P->d_meet;
        ce = cudaMemcpyAsync((void*)a.path_off, P->path_off.data(), (NQ + 1) * 8, cudaMemcpyHostToDevice,
                             P->stream);
        if (ce != cudaSuccess) {
            cudaGetLastError();
            plan_free_partial(P.get());
            return PPSP_ERR_CUDA;
        }
        P->paths = true;
    }
    *out = P.release();
    return PPSP_OK;
}

static void plan_free(ppsp_plan* P) {
    if (!P) return;
    if (P->host_call)
        ;  // its work has ended (host_finish)
    else if (P->stream)
        cudaStreamSynchronize(P->stream);
    else
        cudaDeviceSynchronize();
    for (Slot* s : P->slots) slot_release(P->g, s);
    if (P->gexec) cudaGraphExecDestroy(P->gexec);
    if (P->d_arena && !P->host_call) cudaFreeAsync(P->d_arena, P->stream);
    if (P->d_paths) cudaFreeAsync(P->d_paths, P->stream);
    cudaGetLastError();
    delete P;
}

static ppsp_status plan_launch_direct(ppsp_plan* P, u64* d_out);

// Capture the launches of one run into a CUDA graph (once per output pointer)
// and replay it; any capture failure falls back to direct launches.
static ppsp_status plan_launch(ppsp_plan* P, u64* d_out) {
    P->last_used_graph = false;
    bool dirty = false;
    for (const Slot* s : P->slots) dirty = dirty || s->dirty;
    if (!P->opt.cuda_graph || P->stream == nullptr || P->graph_failed || dirty)
        return plan_launch_direct(P, d_out);
    if (P->gexec == nullptr || P->gexec_out != d_out) {
        if (P->gexec) {
            cudaGraphExecDestroy(P->gexec);
            P->gexec = nullptr;
        }
        cudaGraph_t graph = nullptr;
        if (cudaStreamBeginCapture(P->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
            cudaGetLastError();
            P->graph_failed = true;
            return plan_launch_direct(P, d_out);
        }
        ppsp_status st = plan_launch_direct(P, d_out);
        cudaError_t ce = cudaStreamEndCapture(P->stream, &graph);
        if (st != PPSP_OK || ce != cudaSuccess || graph == nullptr) {
            cudaGetLastError();
            if (graph) cudaGraphDestroy(graph);
            P->graph_failed = true;
            return plan_launch_direct(P, d_out);
        }
        ce = cudaGraphInstantiate(&P->gexec, graph, 0);
        cudaGraphDestroy(graph);
        if (ce != cudaSuccess) {
            cudaGetLastError();
            P->gexec = nullptr;
            P->graph_failed = true;
            return plan_launch_direct(P, d_out);
        }
        P->gexec_out = d_out;
    }
    PPSP_CUDA_TRY(cudaGraphLaunch(P->gexec, P->stream));
    P->launched = true;
    P->last_used_graph = true;
    return PPSP_OK;
}

static ppsp_status plan_launch_direct(ppsp_plan* P, u64* d_out) {
    for (Slot* s : P->slots) {
        ppsp_status st = slot_scrub(s, P->stream);
        if (st != PPSP_OK) return st;
    }
    ppsp_status st = PPSP_OK;
    if (!P->host_call) PPSP_CUDA_TRY(cudaMemsetAsync(P->d_runstate, 0, P->runstate_bytes, P->stream));
    if (P->paths && !P->qedges.empty())
        PPSP_CUDA_TRY(cudaMemsetAsync(P->d_meet, 0xFF, P->qedges.size() * 4, P->stream));
    if (P->model && !P->groups.empty()) {
        // learned Delta per group, written into the device group descriptors
        st = mlp_launch_infer(P->model, P->d_feats, P->groups.size(), nullptr, const_cast<GroupDev*>(P->args.groups),
                              P->delta_default, P->stream);
        if (st != PPSP_OK) return st;
    }
    if (!P->groups.empty()) {
        st = launch_engine(P->args, P->dist_bits, P->block, P->grid, P->stream, P->kind);
        if (st != PPSP_OK) return st;
    }
    if (d_out) {
        st = launch_scatter(P->d_map, P->args.mu, P->k, d_out, P->stream);
        if (st != PPSP_OK) return st;
    }
    P->launched = true;
    return PPSP_OK;
}

static ppsp_status plan_result(ppsp_plan* P, u32 err, const EngineCounters& ec, ppsp_counters* counters) {
    if (counters) {
        memset(counters, 0, sizeof(*counters));
        counters->extracted = ec.extracted;
        counters->edges = ec.edges;
        counters->relaxed = ec.relaxed;
        counters->pushed = ec.pushed;
        counters->rounds = ec.rounds;
        counters->groups = ec.groups;
        counters->searches = ec.searches;
        counters->touched = ec.touched;
        counters->dense_rounds = ec.dense_rounds;
    }
    if (err) {
        for (Slot* s : P->slots) s->dirty = true;
        if (err & ERRB_OVERFLOW) return PPSP_ERR_OVERFLOW;
        if (err & ERRB_TIMEOUT) return PPSP_ERR_TIMEOUT;
        set_last_device_error(err);
        return PPSP_ERR_CUDA;
    }
    return PPSP_OK;
}

// A call from host pairs to host answers: one copy brings back the error word,
// the counters and mu, one wait ends the call, and the answers are put in input
// order here.  With an output array, a scatter launch, three
// copies and four waits a query on the 64^2 grid took 114 us and a batch of 100
// 334; now 81 and 299.
static ppsp_status host_finish(ppsp_plan* P, ppsp_counters* counters, uint64_t* dists_out) {
    char* h = P->g->ws.host;
    cudaError_t ce = cudaMemcpyAsync(h, (char*)P->d_arena + P->back_at, P->back_bytes, cudaMemcpyDeviceToHost, P->stream);
    const cudaError_t cw = cudaStreamSynchronize(P->stream);
    if (ce == cudaSuccess) ce = cw;
    if (ce != cudaSuccess) {
        set_last_cuda_error(ce, "ppsp_batch", __FILE__, __LINE__);
        cudaGetLastError();
        return PPSP_ERR_CUDA;
    }
    u32 err = 0;
    EngineCounters ec{};
    memcpy(&err, h, 4);
    memcpy(&ec, h + ((const char*)P->args.counters - (const char*)P->args.err), sizeof(ec));
    const ppsp_status st = plan_result(P, err, ec, counters);
    if (st != PPSP_OK) return st;
    const char* mu = h + ((const char*)P->args.mu - (const char*)P->args.err);
    for (u64 q = 0; q < P->k; ++q) {
        u64 d = 0;
        if (P->map[q] != NONE) memcpy(&d, mu + (size_t)P->map[q] * 8, 8);
        dists_out[q] = d;
    }
    return PPSP_OK;
}

static ppsp_status plan_wait(ppsp_plan* P, ppsp_counters* counters) {
    if (P->stream) {
        PPSP_CUDA_TRY(cudaStreamSynchronize(P->stream));
    } else {
        PPSP_CUDA_TRY(cudaDeviceSynchronize());
    }
    u32 err = 0;
    EngineCounters ec{};
    PPSP_CUDA_TRY(cudaMemcpyAsync(&err, P->args.err, 4, cudaMemcpyDeviceToHost, P->stream));
    PPSP_CUDA_TRY(cudaMemcpyAsync(&ec, P->args.counters, sizeof(ec), cudaMemcpyDeviceToHost, P->stream));
    PPSP_CUDA_TRY(cudaStreamSynchronize(P->stream));
    return plan_result(P, err, ec, counters);
}

extern "C" {

ppsp_status ppsp_plan_create(ppsp_graph* g, const uint32_t* pairs, uint64_t k, const ppsp_options* opt,
                             ppsp_plan** out) {
    if (!g || !out) return PPSP_ERR_INVALID_ARG;
    *out = nullptr;
    std::lock_guard<std::mutex> lk(g->mu);
    return plan_create_impl(g, pairs, k, opt, false, out);
}

ppsp_status ppsp_plan_run(ppsp_plan* p, uint64_t* d_dists_out) {
    if (!p) return PPSP_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(p->g->mu);
    return plan_launch(p, d_dists_out);
}

ppsp_status ppsp_plan_sync(ppsp_plan* p, ppsp_counters* counters) {
    if (!p) return PPSP_ERR_INVALID_ARG;
    if (!p->launched) return PPSP_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(p->g->mu);
    return plan_wait(p, counters);
}

ppsp_status ppsp_plan_features(const ppsp_plan* p, float* out, uint64_t cap, uint64_t* ngroups) {
    if (!p || !ngroups) return PPSP_ERR_INVALID_ARG;
    *ngroups = p->groups.size();
    if (out) {
        if (cap < p->groups.size()) return PPSP_ERR_BUFFER_TOO_SMALL;
        memcpy(out, p->feats.data(), p->feats.size() * 4);
    }
    return PPSP_OK;
}

ppsp_status ppsp_plan_group_times(ppsp_plan* p, uint64_t* out_ns, uint64_t cap, uint64_t* ngroups) {
    if (!p || !ngroups) return PPSP_ERR_INVALID_ARG;
    *ngroups = p->groups.size();
    if (!out_ns) return PPSP_OK;
    if (cap < p->groups.size()) return PPSP_ERR_BUFFER_TOO_SMALL;
    if (!p->launched) return PPSP_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(p->g->mu);
    if (p->stream) {
        PPSP_CUDA_TRY(cudaStreamSynchronize(p->stream));
    } else {
        PPSP_CUDA_TRY(cudaDeviceSynchronize());
    }
    if (!p->groups.empty())
        PPSP_CUDA_TRY(cudaMemcpy(out_ns, p->args.group_ns, p->groups.size() * 8, cudaMemcpyDeviceToHost));
    return PPSP_OK;
}

ppsp_status ppsp_batch_sources(const uint32_t* pairs, uint64_t k, int32_t strategy, uint32_t flags,
                               uint32_t* src_out, uint32_t* dir_out, uint64_t* n_sources) {
    if ((k && !pairs) || (k && !src_out) || !n_sources) return PPSP_ERR_INVALID_ARG;
    if (strategy != PPSP_BATCH_SSSP && strategy != PPSP_BATCH_VC) return PPSP_ERR_INVALID_ARG;
    // the same deduplication as the plan: unordered pairs for VC-SSSP on an
    // undirected graph, ordered pairs otherwise
    const bool directed = !(flags & PPSP_UNDIRECTED);
    const bool unordered = !directed && strategy == PPSP_BATCH_VC;
    std::unordered_map<u64, u32> qe_id;
    std::vector<std::pair<u32, u32>> uq;
    std::vector<u32> map(k, NONE);
    for (u64 q = 0; q < k; ++q) {
        const u32 s = pairs[2 * q], t = pairs[2 * q + 1];
        if (s == t) continue;
        const u64 key = unordered ? (((u64)std::min(s, t) << 32) | std::max(s, t)) : (((u64)s << 32) | t);
        auto it = qe_id.find(key);
        if (it == qe_id.end()) {
            it = qe_id.emplace(key, (u32)uq.size()).first;
            uq.emplace_back(s, t);
        }
        map[q] = it->second;
    }
    const std::vector<SrcDir> src = sssp_sources(strategy, directed, uq);
    std::unordered_set<u64> distinct;
    for (const SrcDir& x : src) distinct.insert(((u64)x.v << 1) | x.dir);
    for (u64 q = 0; q < k; ++q) {
        src_out[q] = (map[q] == NONE) ? NONE : src[map[q]].v;
        if (dir_out) dir_out[q] = (map[q] == NONE) ? 0u : src[map[q]].dir;
    }
    *n_sources = distinct.size();
    return PPSP_OK;
}

ppsp_status ppsp_plan_launch_shape(const ppsp_plan* p, ppsp_launch_shape* out) {
    if (!p || !out) return PPSP_ERR_INVALID_ARG;
    *out = ppsp_launch_shape{};
    out->kernel = (int32_t)p->kind;
    out->block_threads = p->block;
    out->ctas = p->grid;
    out->teams = (u32)p->team_size.size();
    out->cluster = std::max<u32>(1, p->args.cluster);
    out->long_groups = p->args.long_ctas ? (u32)p->queue_items[0].size() : 0;
    return PPSP_OK;
}

ppsp_status ppsp_plan_device_bytes(const ppsp_plan* p, uint64_t* slot_bytes, uint64_t* teams,
                                   uint64_t* other_bytes) {
    if (!p) return PPSP_ERR_INVALID_ARG;
    u64 sb = 0;
    for (const Slot* s : p->slots) sb += s->bytes;
    u64 ob = p->arena_bytes;
    if (p->d_paths) {
        const u64 NQ = p->qedges.size();
        auto al = [](u64 x) { return (x + 255) & ~255ull; };
        ob += std::max<u64>(256, al(p->path_off[NQ] * 4) + al((NQ + 1) * 8) + al(NQ * 8) + al(NQ * 4));
    }
    if (slot_bytes) *slot_bytes = sb;
    if (teams) *teams = p->slots.size();
    if (other_bytes) *other_bytes = ob;
    return PPSP_OK;
}

ppsp_status ppsp_slot_bytes(const ppsp_graph* g, uint32_t searches, int32_t dist_bits, int32_t frontier,
                            uint64_t* out) {
    if (!g || !out || searches == 0 || searches > (u32)KMAX) return PPSP_ERR_INVALID_ARG;
    if (dist_bits != 32 && dist_bits != 64) return PPSP_ERR_INVALID_ARG;
    if (frontier < PPSP_FRONTIER_AUTO || frontier > PPSP_FRONTIER_DENSE) return PPSP_ERR_INVALID_ARG;
    // the plan's layouts: a group of k searches spans n * 2^ceil(log2 k)
    // interleaved entries (k entries per vertex for pairs and singles)
    const u64 range = (u64)g->n << ceil_log2(searches);
    // the larger touched list of a team that spans the whole grid
    const SlotCaps sc = slot_caps(range, frontier, true);
    *out = slot_alloc_bytes(dist_bits, sc.flat_cap, sc.qcap, sc.tcap);
    return PPSP_OK;
}

ppsp_status ppsp_plan_uses_graph(const ppsp_plan* p, int32_t* out) {
    if (!p || !out) return PPSP_ERR_INVALID_ARG;
    *out = p->last_used_graph ? 1 : 0;
    return PPSP_OK;
}

void ppsp_plan_destroy(ppsp_plan* p) {
    if (!p) return;
    ppsp_graph* g = p->g;
    std::lock_guard<std::mutex> lk(g->mu);
    plan_free(p);
}

struct HostPaths {
    uint32_t* buf = nullptr;          // caller's path buffer
    const uint64_t* offsets = nullptr;  // per query [k+1] (batch), or null (single query)
    uint64_t single_cap = 0;          // single query: capacity
    uint64_t* lens = nullptr;         // per query needed lengths
};

static ppsp_status run_host(ppsp_graph* g, const uint32_t* pairs, uint64_t k, const ppsp_options* opt,
                            bool single, uint64_t* dists_out, ppsp_counters* counters, const HostPaths* hp) {
    ppsp_plan* P = nullptr;
    std::vector<u64> caps;
    if (hp) {
        caps.resize(k);
        for (u64 q = 0; q < k; ++q) caps[q] = hp->offsets ? hp->offsets[q + 1] - hp->offsets[q] : hp->single_cap;
    }
    ppsp_status st = plan_create_impl(g, pairs, k, opt, single, &P, hp ? caps.data() : nullptr, true);
    if (st != PPSP_OK) {
        g->ws.trim(opt ? (cudaStream_t)opt->stream : nullptr);
        return st;
    }
    st = plan_launch_direct(P, nullptr);
    if (st == PPSP_OK)
        st = host_finish(P, counters, dists_out);
    else
        cudaStreamSynchronize(P->stream);
    cudaError_t ce = cudaSuccess;
    if (st == PPSP_OK && hp && P->paths) {
        // device paths are per query edge, oriented from its first to its
        // second endpoint; copy (or reverse) them into each query's slice
        const u64 NQ = P->qedges.size();
        std::vector<u64> plen(NQ, 0);
        std::vector<u32> pbuf(P->path_off[NQ]);
        if (NQ) {
            ce = cudaMemcpyAsync(plen.data(), P->args.path_len, NQ * 8, cudaMemcpyDeviceToHost, P->stream);
            if (ce == cudaSuccess && !pbuf.empty())
                ce = cudaMemcpyAsync(pbuf.data(), P->args.path_buf, pbuf.size() * 4, cudaMemcpyDeviceToHost,
                                     P->stream);
            if (ce == cudaSuccess) ce = cudaStreamSynchronize(P->stream);
            if (ce != cudaSuccess) {
                cudaGetLastError();
                st = PPSP_ERR_CUDA;
            }
        }
        bool small = false;
        for (u64 q = 0; q < k && st == PPSP_OK; ++q) {
            const u32 s = pairs[2 * q], t = pairs[2 * q + 1];
            uint32_t* dst = hp->buf + (hp->offsets ? hp->offsets[q] : 0);
            const u64 cap = caps[q];
            u64 len = 0;
            if (s == t) {
                len = 1;
                if (cap >= 1 && hp->buf) dst[0] = s;
            } else if (dists_out[q] != PPSP_INF) {
                const u32 qe = P->map[q];
                len = plen[qe];
                if (len <= cap && len <= P->path_off[qe + 1] - P->path_off[qe] && hp->buf) {
                    // device ids back to the caller's
                    const u32* src = pbuf.data() + P->path_off[qe];
                    const u32 s_dev = g->perm.empty() ? s : g->perm[s];
                    const bool fwd = (P->qedge_ends[qe].first == s_dev);
                    for (u64 x = 0; x < len; ++x) {
                        const u32 y = fwd ? src[x] : src[len - 1 - x];
                        dst[x] = g->inv.empty() ? y : g->inv[y];
                    }
                } else {
                    small = true;
                }
            }
            if (hp->lens) hp->lens[q] = len;
        }
        if (st == PPSP_OK && small) st = PPSP_ERR_BUFFER_TOO_SMALL;
    }
    plan_free(P);
    g->ws.trim(opt ? (cudaStream_t)opt->stream : nullptr);
    return st;
}

ppsp_status ppsp_query(ppsp_graph* g, uint32_t s, uint32_t t, const ppsp_options* opt, uint64_t* dist_out,
                       uint32_t* path_buf, uint64_t path_cap, uint64_t* path_len) {
    if (!g || !dist_out) return PPSP_ERR_INVALID_ARG;
    if (path_len) *path_len = 0;
    uint32_t pr[2] = {s, t};
    std::lock_guard<std::mutex> lk(g->mu);
    if (opt && opt->want_paths) {
        if (path_cap && !path_buf) return PPSP_ERR_INVALID_ARG;
        HostPaths hp;
        hp.buf = path_buf;
        hp.single_cap = path_cap;
        hp.lens = path_len;
        return run_host(g, pr, 1, opt, true, dist_out, nullptr, &hp);
    }
    return run_host(g, pr, 1, opt, true, dist_out, nullptr, nullptr);
}

ppsp_status ppsp_batch(ppsp_graph* g, const uint32_t* pairs, uint64_t k, const ppsp_options* opt,
                       uint64_t* dists_out, uint32_t* paths_buf, const uint64_t* path_offsets, uint64_t* path_lens,
                       ppsp_counters* counters) {
    if (!g || (k && (!pairs || !dists_out))) return PPSP_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(g->mu);
    if (opt && opt->want_paths) {
        if (k && (!path_offsets || !paths_buf)) return PPSP_ERR_INVALID_ARG;
        for (u64 q = 0; q < k; ++q)
            if (path_offsets[q + 1] < path_offsets[q]) return PPSP_ERR_INVALID_ARG;
        HostPaths hp;
        hp.buf = paths_buf;
        hp.offsets = path_offsets;
        hp.lens = path_lens;
        return run_host(g, pairs, k, opt, false, dists_out, counters, &hp);
    }
    return run_host(g, pairs, k, opt, false, dists_out, counters, nullptr);
}

}  // extern "C"

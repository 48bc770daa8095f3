// Bucketed search kernel for graphs of low degree (road and grid shapes): one
// CTA, or a cluster of them (see bk_gather), runs a group of one or two
// searches to completion, and a team of CTAs a Multi-BiDS group, one search
// each (see bk_update).
//
// Same algorithm as run_local (engine_core.cuh): Delta*-stepping buckets in
// shared memory with lazy deletion, a far list beyond the ring's window, a
// spill bitmap as the last resort.  What differs is the work of one step,
// which on these graphs is short (100 to 500 entries) and bound by the chain
// of dependent accesses and by instruction issue, not by bandwidth:
//
//  * Adjacency blocks: the first four edges of vertex v lie in one aligned
//    block (GraphDev::blk16 / blk8: 64 bytes with the targets' potential
//    coordinates, 32 without), so an entry needs neither its offsets nor a
//    prefix sum over degrees: four lanes take one entry, lane q its q-th edge,
//    and the block and the entry's distance are loaded together.  The chain is
//    ring entry -> {block, own distance} -> target distance.  A vertex of more
//    than four edges is inserted as two entries, so its continued edges are
//    another entry's work, not a second pass of the same warp.
//  * No potential at extraction: an entry's prune value is known from its
//    bucket to within one step, and the stop rule (bk_decide) compares the
//    bucket's smallest prune value with the bound, so testing each entry again
//    would only save part of the last bucket.  The rule subtracts the key
//    offset (h(s, t) for BiD-A*), which run_local's does not: it stops about
//    12% of the steps earlier on the 1024^2 road graph.
//  * The bucket index comes from a multiplication by a rounded-down reciprocal
//    of the step, which gives the exact bucket or the one before it: an entry
//    may be taken one step early, never late, and (b - 1) * step stays a lower
//    bound of the keys in bucket b.
//  * Positions in a bucket come from plain shared-memory atomics (78 cycles
//    for 32 lanes on one address; a match of the lanes by bucket takes 99
//    before its own atomic).
//
// Measured against run_local (which took 17,000 cycles a step for one query
// alone on the GPU: decision 3,400, extraction 4,100, relaxation 6,900, the
// rest waiting; an L2 hit takes 290-360): one BiD-A* query on the 1024^2 road
// graph 7.3 -> 2.4 ms (4.6 -> 1.1 ms over random pairs, where the queue path
// took the whole GPU), 1,000 queries on it 45.5 -> 16.4 ms, 2,048 on the 2048^2
// graph 228 -> 100 ms, 256 with 64-bit distances on the 4096^2 graph 255 ->
// 136 ms.  With the longest pairs on more threads beside the rest (long_groups
// in plan.cu) the 1,000 take 12.7 ms and the 256 82 to 93.  DRAM traffic of the
// 2,048: 383 -> 213 GB.  What bounds it now: per
// step and active warp about 500 instructions at 12.6 cycles each, of which a
// third waits on global loads, a fifth on fixed-latency results and a seventh
// on shared memory (one query alone); on a full GPU 0.46 of the issue slots
// and 2.1 TB/s of random sectors, of the 1.95 TB/s that 155,000 independent
// 4-byte loads from 1 GB reach.  Collecting the successful relaxations of the
// CTA in shared memory, so that full warps take the second half, cut the
// instructions but added a barrier per pass: 2,048 queries 100 -> 131 ms.
#pragma once

#include "engine_core.cuh"

namespace ppsp {

constexpr u32 BK_NB = 64;      // buckets in the ring (a power of two, two per lane of the deciding warp)
constexpr u32 BK_DEFER = 64;   // entries with many edges handed to the whole CTA, per step
constexpr u32 BK_QUAD_MAX = 32;  // continued edges that an entry's four lanes scan themselves
constexpr u32 BK_EXTRA = 1u << 31;  // of a ring entry: the vertex's continued edges; of a target: it has some

// Compiled variants: BiDS and BiD-A* pairs, single searches (ET, A*, SSSP),
// which tell their mode apart at run time, and one search of a Multi-BiDS
// group.  The last two are one search: their ring and lists hold vertices.
enum { BK_BIDS = 0, BK_BIDASTAR = 1, BK_SINGLE = 2, BK_MULTI = 3 };
constexpr bool bk_one(int kind) { return kind == BK_SINGLE || kind == BK_MULTI; }

// How a group of one or two searches is run, and the kernel's instances: by
// one CTA; the same, with teams of CTAs for the larger groups; by a cluster.
enum { BK_CTAS = 0, BK_TEAMS = 1, BK_CLUSTERS = 2 };
constexpr u32 BK_CL_MAX = 8;  // CTAs of a cluster (the portable limit)

// What the CTAs of a cluster tell each other at the end of a step.
struct BkPub {
    u64 far_min, bound;
    u32 far_n, full, late, spill, fresh, cnt0, cnt1, pad;
    u32 rn[BK_NB];
};

struct BkShared {
    // the decision of a step, read by every thread
    u64 cur, curkey;      // the bucket of the step and its threshold cur * step
    u32 what, n, slot;    // what: 0 process bucket cur, 1 re-bucket far, 2 recover spills, 3 done
    u32 late;             // 1 + largest (curkey - key) of the step's late entries, 0: none
    u64 bound;            // prune bound: mu, or the largest target distance (SSSP)
    u64 step;
    i64 key_off;          // added to prune values to give keys (one value per group)
    int2 pa, pb;          // anchors of search 0's potential: h_pb - h_pa (A*: h_pb)
    u32 rn[BK_NB];
    // far list: entries, smallest bucket, which of the slot's two arrays, and
    // the entries right after the last re-bucketing
    u32 far_n, far_at, far_after;
    u64 far_min;
    u32 tn, tov, spill, recov, idle;
    u32 cnt_dir[2];       // stored entries per direction (pairs, kept while mu is unset)
    u32 ndef;
    SlotDev dev;          // the slot (its arrays are indexed at run time)
    u32 src[2], sdir[2], pcnt[2];
    PartnerDev pcache[2];
    u32 group, flag;
    // clusters: published states (two in turn), and the entries that CTAs 0 ..
    // r - 1 hold of the step's bucket; this CTA takes entries e0 .. n - 1 of all
    BkPub pub[2];
    u32 pre[BK_CL_MAX + 1], e0, any_spill;
    // a Multi-BiDS search: its partners j, their query edges and mu (mirrors,
    // never below a.mu); muj[j] = 0 where j is no partner
    u32 pj[KMAX], npart;
    u32 qej[KMAX];
    u64 muj[KMAX];
    u32 def_at[BK_DEFER], def_cnt[BK_DEFER], def_f[BK_DEFER];
    u64 def_d[BK_DEFER];
};

__device__ __forceinline__ PartnerDev partner(const EngineArgs&, const BkShared& sm, u32 i, u32) { return sm.pcache[i]; }

// A ring entry: flat index (BK_EXTRA), distance at insertion.
template <typename D>
struct BkEntry;
template <>
struct BkEntry<u32> {
    typedef uint2 T;
    static __device__ __forceinline__ T make(u32 f, u64 d) { return make_uint2(f, (u32)d); }
};
template <>
struct BkEntry<u64> {
    typedef ulonglong2 T;
    static __device__ __forceinline__ T make(u32 f, u64 d) { return make_ulonglong2(f, d); }
};

template <typename D>
constexpr size_t bucket_smem_bytes(u32 cap) {
    return ((sizeof(BkShared) + 15) & ~(size_t)15) + (size_t)BK_NB * cap * sizeof(typename BkEntry<D>::T);
}

// One group's view: everything the inner functions need, in registers.
template <typename D>
struct BkCtx {
    D* dist;
    u32* touched;
    typename BkEntry<D>::T* ring;
    u32 cap, ob;  // shared-memory entries per bucket, entries of its overflow region
    u32 tcap;
    u32 mode, target, qe;
    u32 d0, dm;   // direction of search i: d0 | (i & dm)
    u32 cl, rank; // cluster: its CTAs and this one's place
    u32 ks, i0;   // one search of a group: its distances are dist[(v << ks) | i0]
    u32 magic;    // floor(2^32 / step)
    u32 cur_lo;   // this step's bucket (low bits)
    i64 kc;       // the group's key offset less that threshold: key - threshold = prune value + kc
    u32 c_x, c_e, c_r, c_p, c_t;
    int dc0, dc1;  // net change of the per-direction entry counts (pairs)
};

// mu <- min(mu, s); s is the length of a real path.
template <typename D>
__device__ __forceinline__ void bk_try_mu(const EngineArgs& a, const BkCtx<D>& c, BkShared& sm, u64 s) {
    if (s >= sm.bound) return;
    atomicMin(reinterpret_cast<unsigned long long*>(&sm.bound), (unsigned long long)s);
    atomicMin(reinterpret_cast<unsigned long long*>(a.mu + c.qe), (unsigned long long)s);
}

// h_x(v) = floor(|P(v) - P(x)| / 2^F), exact: r with (r 2^F)^2 <= |P(v) - P(x)|^2
// < ((r + 1) 2^F)^2, from a float32 estimate and integer comparisons.  The
// estimate's relative error is below 2^-21 (the roundings of the differences,
// the sum and the hardware root), a few units below 2^24; above, float64.
// Coordinates are below 2^30 in magnitude, so differences fit 32 bits and the
// square of (r + 1) 2^F 64.
__device__ __forceinline__ float bk_h_est(int dx, int dy, float scale) {
    const float fx = (float)dx, fy = (float)dy;
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(fx * fx + fy * fy));
    return y * scale;
}
static __device__ __noinline__ u64 bk_h_big(u64 d2, u32 shift) { return (u64)sqrt((double)d2) >> shift; }
__device__ __forceinline__ u32 bk_h_fix(int dx, int dy, float est, u32 shift) {
    const u64 d2 = (u64)((i64)dx * dx) + (u64)((i64)dy * dy);
    const u32 one = 1u << shift;
    u32 R = (est < 16777216.f ? (u32)est : (u32)bk_h_big(d2, shift)) << shift;
    while ((u64)R * R > d2) R -= one;
    while ((u64)(R + one) * (R + one) <= d2) R += one;
    return R >> shift;
}

// Prune value of <v, i> at distance d (Table 2); q = P(v).
template <typename D, int KIND>
__device__ __forceinline__ i64 bk_prune_value(const EngineArgs& a, const BkCtx<D>& c, const BkShared& sm, u32 i,
                                              int2 q, u64 d) {
    if (KIND == BK_BIDS || KIND == BK_MULTI) return 2 * (i64)d;
    if (KIND == BK_SINGLE && c.mode != GM_ASTAR) return (i64)d;
    const u32 F = a.g.pot_shift;
    const float scale = __uint_as_float((127u - F) << 23);  // 2^-F
    const int2 pb = sm.pb;
    const int bx = q.x - pb.x, by = q.y - pb.y;
    const float eb = bk_h_est(bx, by, scale);
    if (KIND == BK_SINGLE) return (i64)d + (i64)bk_h_fix(bx, by, eb, F);
    const int2 pa = sm.pa;
    const int ax = q.x - pa.x, ay = q.y - pa.y;
    const float ea = bk_h_est(ax, ay, scale);
    const i64 rho = (i64)bk_h_fix(bx, by, eb, F) - (i64)bk_h_fix(ax, ay, ea, F);
    return 2 * (i64)d + (i ? -rho : rho);
}

// Entry (f, d) at position pos of ring slot s: shared memory, then the
// bucket's overflow region.
template <typename D>
__device__ __forceinline__ bool bk_place(const BkCtx<D>& c, const BkShared& sm, u32 s, u32 pos, u32 f, u64 d) {
    if (pos < c.cap) {
        c.ring[s * c.cap + pos] = BkEntry<D>::make(f, d);
        return true;
    }
    pos -= c.cap;
    if (pos >= c.ob) return false;
    sm.dev.of[(size_t)s * c.ob + pos] = f;
    reinterpret_cast<D*>(sm.dev.od)[(size_t)s * c.ob + pos] = (D)d;
    return true;
}

template <typename D>
__device__ __forceinline__ bool bk_place_far(const BkShared& sm, u32 fb, u32 pos, u32 f, u64 d) {
    if (pos >= sm.dev.qcap) return false;
    sm.dev.q[fb][pos] = f;
    reinterpret_cast<D*>(sm.dev.fd[fb])[pos] = (D)d;
    return true;
}

// An entry that found no room: its bit in the slot's spill bitmap.  It is
// recovered later with both parts (and counted as another entry; a part that
// was stored is then taken twice, which is harmless).  Returns 1 for a new bit.
static __device__ __noinline__ u32 bk_spill(BkShared& sm, u32 f) {
    const u32 bit = 1u << (f & 31u);
    if (atomicOr(sm.dev.bm[0] + (f >> 5), bit) & bit) return 0;
    sm.spill = 1;
    return 1;
}

// Far entries: beyond the ring's window.
template <typename D>
__device__ __forceinline__ void bk_insert_far(BkShared& sm, u32 db, u32 f, u32 f0, u32 num, u64 d, bool& s0, bool& s1) {
    const u32 pos = atomicAdd(&sm.far_n, num);
    s0 = bk_place_far<D>(sm, sm.far_at, pos, f0, d);
    if (num == 2) s1 = bk_place_far<D>(sm, sm.far_at, pos + 1, f | BK_EXTRA, d);
    atomicMin(reinterpret_cast<unsigned long long*>(&sm.far_min), (unsigned long long)(sm.cur + db));
}

// F.Add of flat index f at distance d and prune value pv.  extra: 0 its first
// edges, BK_EXTRA its continued ones, 2 both (two entries).
template <typename D, int KIND>
__device__ __forceinline__ void bk_insert(BkCtx<D>& c, BkShared& sm, u32 f, u32 extra, i64 pv, u64 d) {
    const i64 rk = pv + c.kc;  // key less the step's threshold
    const u32 num = extra == 2 ? 2u : 1u, f0 = extra == BK_EXTRA ? (f | BK_EXTRA) : f;
    u32 db;  // buckets ahead of the current one
    if (rk <= 0) {
        // already under the threshold: due at the next step; the bucket's
        // lower bound does not hold for it, so its distance below the
        // threshold is remembered
        db = 1;
        const u64 below = (u64)-rk + 1;
        atomicMax(&sm.late, below >> 32 ? 0xFFFFFFFFu : (u32)below);
    } else if (((u64)rk >> 32) == 0) {
        db = __umulhi((u32)rk - 1u, c.magic) + 1u;
    } else {
        const u64 q = ((u64)rk - 1) / sm.step + 1;
        db = q < 0x7FFFFFFFull ? (u32)q : 0x7FFFFFFFu;
    }
    bool s0, s1 = true;  // stored: the entry, and its second one
    if (db < BK_NB) {
        const u32 s = (c.cur_lo + db) & (BK_NB - 1);
        const u32 pos = atomicAdd(&sm.rn[s], num);
        s0 = bk_place<D>(c, sm, s, pos, f0, d);
        if (num == 2) s1 = bk_place<D>(c, sm, s, pos + 1, f | BK_EXTRA, d);
    } else {
        bk_insert_far<D>(sm, db, f, f0, num, d, s0, s1);
    }
    ++c.c_p;
    u32 num_in = (s0 && extra != BK_EXTRA) ? 1u : 0u;  // stored entries that count for their direction
    if (!(s0 && s1)) num_in += bk_spill(sm, f);
    if (!bk_one(KIND)) {
        if (f & 1u) c.dc1 += num_in; else c.dc0 += num_in;
    }
}

// The distance of <v, i> and, in a pair, the other search's (in the slot's
// width: 64-bit copies of 32-bit distances cost registers and instructions).
template <typename D, int KIND>
__device__ __forceinline__ void bk_load(const BkCtx<D>& c, u32 v, u32 i, D& own, D& oth) {
    if (!bk_one(KIND)) {
        u64 x0, x1;
        ld_pair(c.dist, v, x0, x1);
        own = (D)(i ? x1 : x0);
        oth = (D)(i ? x0 : x1);
    } else {
        own = (D)ld_dist(c.dist + (KIND == BK_MULTI ? (((size_t)v << c.ks) | c.i0) : (size_t)v));
        oth = (D)DT<D>::INF;
    }
}

// Address of the distance of flat index f.
template <typename D, int KIND>
__device__ __forceinline__ D* bk_at(const BkCtx<D>& c, u32 f) {
    return c.dist + (KIND == BK_MULTI ? (((size_t)f << c.ks) | c.i0) : (size_t)f);
}

// UpdateDistance of a Multi-BiDS search at vertex v, whose distance nd it has
// just written.  The searches of a group run on CTAs of their own with no
// barrier between them (each at its own threshold: Theorem 3.3 holds per query
// for any schedule, and their frontiers grow at about the same rate).  Two
// searches that write their final distances of v at the same time must not
// miss each other: each writes with an atomic whose result it waits for, then
// a fence, then reads the other's distance, so whichever write comes second
// sees the first.  Nothing has to be read again at extraction.
//
// Measured (24-clique on the 1024^2 road graph, 11.8 M extractions): one team
// of all CTAs on the queue / bitmap frontier, which inserts every waiting
// entry again at every step, 244 ms; one CTA per search 41 ms at the same
// increment (48 before the row's loads were issued together; the fence is 8%
// of it), 18.8 ms at the one the model now gives.  Bound by the latency of a
// step whose distances are a 128-byte row apart.
template <typename D>
__device__ __forceinline__ void bk_update_one(const EngineArgs& a, BkShared& sm, u32 j, u64 o, u64 nd) {
    const u64 s = nd + o;
    if (o != DT<D>::INF && s < sm.muj[j]) {
        atomicMin(reinterpret_cast<unsigned long long*>(&sm.muj[j]), (unsigned long long)s);
        atomicMin(reinterpret_cast<unsigned long long*>(a.mu + sm.qej[j]), (unsigned long long)s);
    }
}
template <typename D>
__device__ __forceinline__ void bk_update(const EngineArgs& a, const BkCtx<D>& c, BkShared& sm, u32 v, u64 nd) {
    __threadfence();
    const D* row = c.dist + ((size_t)v << c.ks);
    const u32 np = sm.npart;
    if (np <= 4) {
        for (u32 p = 0; p < np; ++p) bk_update_one<D>(a, sm, sm.pj[p], ld_dist(row + sm.pj[p]), nd);
        return;
    }
    // the whole row, 64 bytes in flight (32: 20.4 instead of 18.8 ms for the
    // clique above); most entries are still infinite
    constexpr u32 V = 16 / sizeof(D), CH = 4;
    for (u32 j0 = 0; j0 < (1u << c.ks); j0 += CH * V) {
        uint4 x[CH];
#pragma unroll
        for (u32 k = 0; k < CH; ++k) {
            x[k] = make_uint4(~0u, ~0u, ~0u, ~0u);
            if (j0 + k * V < (1u << c.ks)) x[k] = __ldcg(reinterpret_cast<const uint4*>(row + j0 + k * V));
        }
#pragma unroll
        for (u32 k = 0; k < CH; ++k) {
            const u32 j = j0 + k * V;
            if ((x[k].x & x[k].y & x[k].z & x[k].w) == ~0u) continue;
            if (sizeof(D) == 4) {
                bk_update_one<D>(a, sm, j, x[k].x, nd);
                bk_update_one<D>(a, sm, j + 1, x[k].y, nd);
                bk_update_one<D>(a, sm, j + 2, x[k].z, nd);
                bk_update_one<D>(a, sm, j + 3, x[k].w, nd);
            } else {
                bk_update_one<D>(a, sm, j, ((u64)x[k].y << 32) | x[k].x, nd);
                bk_update_one<D>(a, sm, j + 1, ((u64)x[k].w << 32) | x[k].z, nd);
            }
        }
    }
}

// Refresh a Multi-BiDS search's mirrors of mu and its prune bound, the
// largest of them (mumax, Table 2), by one warp.
__device__ __forceinline__ void bk_refresh(const EngineArgs& a, BkShared& sm) {
    u64 m = 0;
    for (u32 p = threadIdx.x & 31u; p < sm.npart; p += 32) {
        const u32 j = sm.pj[p];
        const u64 x = ldcg64(a.mu + sm.qej[j]);
        atomicMin(reinterpret_cast<unsigned long long*>(&sm.muj[j]), (unsigned long long)x);
        m = x > m ? x : m;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const u64 y = __shfl_xor_sync(0xffffffffu, m, o);
        m = y > m ? y : m;
    }
    if ((threadIdx.x & 31u) == 0) atomicMin(reinterpret_cast<unsigned long long*>(&sm.bound), (unsigned long long)m);
}

struct BkRec {
    u32 v, w;  // target (bit 31: it has continued edges), weight
    int2 q;    // P(target)
};

// Record k of the adjacency blocks (or, at >= 4n, of the continued edges).
template <int KIND>
__device__ __forceinline__ BkRec bk_rec(const EngineArgs& a, bool pot, u32 dir, size_t k) {
    BkRec r;
    if (KIND == BK_BIDASTAR || (KIND == BK_SINGLE && pot)) {
        const int4 x = __ldg((dir ? a.g.blk16_t : a.g.blk16) + k);
        r.v = (u32)x.x;
        r.w = (u32)x.y;
        r.q = make_int2(x.z, x.w);
    } else {
        const uint2 x = __ldg((dir ? a.g.blk8_t : a.g.blk8) + k);
        r.v = x.x;
        r.w = x.y;
        r.q = make_int2(0, 0);
    }
    return r;
}

// Relaxation along record r of entry <f, d>, given the target's distances
// just read: they decide success (a concurrent smaller write only leaves a
// stale entry behind, which extraction drops), so the write is not waited for.
template <typename D, int KIND>
__device__ __forceinline__ void bk_relax(const EngineArgs& a, BkCtx<D>& c, BkShared& sm, u32 f, D d, const BkRec& r,
                                         D own, D oth) {
    constexpr u32 KS = bk_one(KIND) ? 0u : 1u;
    const u32 i = KS ? (f & 1u) : 0u;
    const D nd = d + (D)r.w;
    ++c.c_e;
    if (nd > (D)DT<D>::MAXV || nd < d) {
        // a distance that does not fit, unless the entry should have been
        // pruned (extraction does not test that)
        const int2 qv = a.g.pc ? __ldg(a.g.pc + (f >> KS)) : make_int2(0, 0);
        if (!pruned(bk_prune_value<D, KIND>(a, c, sm, i, qv, d), sm.bound)) atomicOr(a.err, ERRB_OVERFLOW);
        return;
    }
    if (nd >= own) return;
    const u32 v2 = r.v & ~BK_EXTRA, f2 = (v2 << KS) | i;
    if (KIND == BK_MULTI) {
        if (amin_dist(bk_at<D, KIND>(c, f2), nd) <= (u64)nd) return;
        bk_update<D>(a, c, sm, v2, nd);
    } else {
        amin_dist(c.dist + f2, nd);
    }
    ++c.c_r;
    // the position in the touched list is asked for here and used at the end
    const bool fresh = own == (D)DT<D>::INF;
    u32 tpos = 0;
    if (fresh) {
        ++c.c_t;
        tpos = atomicAdd(&sm.tn, 1u);
    }
    if (!bk_one(KIND)) {
        if (oth != (D)DT<D>::INF) bk_try_mu<D>(a, c, sm, (u64)nd + oth);
    } else if (KIND == BK_SINGLE && v2 == c.target) {
        bk_try_mu<D>(a, c, sm, nd);
    }
    const i64 pv = bk_prune_value<D, KIND>(a, c, sm, i, r.q, nd);
    if (!pruned(pv, sm.bound)) bk_insert<D, KIND>(c, sm, f2, (r.v & BK_EXTRA) ? 2u : 0u, pv, nd);
    if (fresh) {
        if (tpos < c.tcap)
            c.touched[tpos] = f2;
        else
            sm.tov = 1;
    }
}

// Take the bucket's entries: four lanes each.
template <typename D, int B, int KIND, bool CL>
__device__ __forceinline__ void bk_process(const EngineArgs& a, BkCtx<D>& c, BkShared& sm, bool pot) {
    constexpr u32 KS = bk_one(KIND) ? 0u : 1u;
    const u32 t = threadIdx.x, q4 = t & 3u;
    const u32 n = sm.n, s = sm.slot;
    for (u32 e1 = (CL ? sm.e0 : 0u) + (t >> 2); e1 < n; e1 += B / 4) {
        u32 f, e = e1;
        D dins;
        const typename BkEntry<D>::T* ring = c.ring;
        i64 ovf = (i64)((size_t)s * c.ob);
        if (CL) {
            // the entry's holder: its shared memory and its overflow region
            u32 r = 0;
            while (e1 >= sm.pre[r + 1]) ++r;
            e = e1 - sm.pre[r];
            ring = cg::this_cluster().map_shared_rank(c.ring, r);
            ovf += ((i64)r - (i64)c.rank) * (i64)sm.dev.ocap;
        }
        if (e < c.cap) {
            const typename BkEntry<D>::T x = ring[s * c.cap + e];
            f = (u32)x.x;
            dins = (D)x.y;
        } else {
            f = __ldcg(sm.dev.of + ovf + (e - c.cap));
            dins = (D)ld_dist(reinterpret_cast<const D*>(sm.dev.od) + ovf + (e - c.cap));
        }
        const u32 extra = f & BK_EXTRA;
        f &= ~BK_EXTRA;
        const u32 v = f >> KS, i = KS ? (f & 1u) : 0u, dir = c.d0 | (i & c.dm);
        D d, oth;
        bk_load<D, KIND>(c, v, i, d, oth);
        u32 rest = 0;   // continued edges after these four
        size_t at = (size_t)v * 4 + q4;
        if (extra) {
            // the fourth record holds where the edges go on
            at = (size_t)bk_rec<KIND>(a, pot, dir, (size_t)v * 4 + 3).w + q4;
            const u32* off = dir ? a.g.off_t : a.g.off;
            rest = __ldg(off + v + 1) - __ldg(off + v) - 3;
            rest = rest > 4 ? rest - 4 : 0;
        }
        BkRec r = bk_rec<KIND>(a, pot, dir, at);
        if (!bk_one(KIND) && q4 == 0 && !extra) {
            if (i) --c.dc1; else --c.dc0;  // the stored entry is consumed
        }
        if (d != dins) continue;  // stale: a smaller distance was inserted again
        if (q4 == 0 && !extra) {
            ++c.c_x;
            if (!bk_one(KIND) && oth != (D)DT<D>::INF) bk_try_mu<D>(a, c, sm, (u64)d + oth);
        }
        if (r.v < BLK_MORE) {
            D own;
            bk_load<D, KIND>(c, r.v & ~BK_EXTRA, i, own, oth);
            bk_relax<D, KIND>(a, c, sm, f, d, r, own, oth);
        }
        if (rest) {
            bool mine = true;
            if (rest > BK_QUAD_MAX) {
                // many edges: for the whole CTA, after the step's barrier
                // (ndef may pass BK_DEFER: the readers clamp it)
                if (q4 == 0) {
                    const u32 k = atomicAdd(&sm.ndef, 1u);
                    if (k < BK_DEFER) {
                        sm.def_at[k] = (u32)(at + 4);
                        sm.def_cnt[k] = rest;
                        sm.def_f[k] = f;
                        sm.def_d[k] = d;
                    } else {
                        // no room: this lane scans them all
                        for (u32 j = 0; j < rest; ++j) {
                            r = bk_rec<KIND>(a, pot, dir, at + 4 + j);
                            D own;
                            bk_load<D, KIND>(c, r.v & ~BK_EXTRA, i, own, oth);
                            bk_relax<D, KIND>(a, c, sm, f, d, r, own, oth);
                        }
                    }
                }
                mine = false;
            }
            for (u32 j = q4; mine && j < rest; j += 4) {
                at += 4;
                r = bk_rec<KIND>(a, pot, dir, at);
                D own;
                bk_load<D, KIND>(c, r.v & ~BK_EXTRA, i, own, oth);
                bk_relax<D, KIND>(a, c, sm, f, d, r, own, oth);
            }
        }
    }
}

// Entries with many edges: the whole CTA shares each one's.
template <typename D, int B, int KIND>
__device__ __forceinline__ void bk_deferred(const EngineArgs& a, BkCtx<D>& c, BkShared& sm, bool pot) {
    const u32 nd = min(sm.ndef, BK_DEFER);
    for (u32 k = 0; k < nd; ++k) {
        const u32 f = sm.def_f[k], i = bk_one(KIND) ? 0u : (f & 1u);
        const D d = (D)sm.def_d[k];
        for (u32 j = threadIdx.x; j < sm.def_cnt[k]; j += B) {
            const BkRec r = bk_rec<KIND>(a, pot, c.d0 | (i & c.dm), (size_t)sm.def_at[k] + j);
            D own, oth;
            bk_load<D, KIND>(c, r.v & ~BK_EXTRA, i, own, oth);
            bk_relax<D, KIND>(a, c, sm, f, d, r, own, oth);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) sm.ndef = 0;
}

// A far or spilled entry back into the ring (or the other far list): dropped
// when stale (dins = INF: a spilled one, taken from its current distance with
// both parts).
template <typename D, int KIND>
__device__ __forceinline__ void bk_rebucket(const EngineArgs& a, BkCtx<D>& c, BkShared& sm, bool pot, u32 f,
                                            u64 dins) {
    constexpr u32 KS = bk_one(KIND) ? 0u : 1u;
    u32 extra = f & BK_EXTRA;
    f &= ~BK_EXTRA;
    const u32 v = f >> KS, i = KS ? (f & 1u) : 0u;
    const u64 d = ld_dist(bk_at<D, KIND>(c, f));
    const int2 q = pot ? __ldg(a.g.pc + v) : make_int2(0, 0);
    if (!bk_one(KIND) && !extra) {
        if (i) --c.dc1; else --c.dc0;
    }
    if (d == DT<D>::INF || (dins != DT<D>::INF && d != dins)) return;
    if (dins == DT<D>::INF) {
        const u32* off = (c.d0 | (i & c.dm)) ? a.g.off_t : a.g.off;
        if (__ldg(off + v + 1) - __ldg(off + v) > 4) extra = 2;
    }
    bk_insert<D, KIND>(c, sm, f, extra, bk_prune_value<D, KIND>(a, c, sm, i, q, d), d);
}

template <typename D, int B, int KIND>
__device__ __forceinline__ void bk_redistribute(const EngineArgs& a, BkCtx<D>& c, BkShared& sm, bool pot) {
    const u32 t = threadIdx.x, from = sm.far_at;
    const u32 n = min(sm.far_n, sm.dev.qcap);
    __syncthreads();
    if (t == 0) {
        sm.far_at = from ^ 1u;
        sm.far_n = 0;
        sm.far_min = INF64;
    }
    __syncthreads();
    for (u32 k = t; k < n; k += B)
        bk_rebucket<D, KIND>(a, c, sm, pot, __ldcg(sm.dev.q[from] + k),
                             ld_dist(reinterpret_cast<const D*>(sm.dev.fd[from]) + k));
    __syncthreads();
    if (t == 0) sm.far_after = sm.far_n;
}

template <typename D, int B, int KIND>
__device__ __forceinline__ void bk_recover(const EngineArgs& a, BkCtx<D>& c, BkShared& sm, bool pot, u32 nwords) {
    if (threadIdx.x == 0) sm.spill = 0;
    __syncthreads();
    for (u32 w = c.rank * B + threadIdx.x; w < nwords; w += c.cl * B) {
        u32 bits = __ldcg(sm.dev.bm[0] + w);
        if (!bits) continue;
        // cleared before its entries are inserted again: one that spills once
        // more sets its bit again
        atomicAnd(sm.dev.bm[0] + w, ~bits);
        while (bits) {
            const u32 f = (w << 5) | (u32)(__ffs(bits) - 1);
            bits &= bits - 1;
            bk_rebucket<D, KIND>(a, c, sm, pot, f, DT<D>::INF);
        }
    }
}

// A cluster runs one group: relaxed entries go to the ring of the CTA that
// relaxed them, and a step takes the bucket's entries of all rings, split
// evenly (read through distributed shared memory).  Each CTA publishes its
// state at the end of a step, the cluster meets at one hardware barrier, and
// every CTA makes the same decision from all states.  A step gains a barrier
// (400-600 cycles) and the reads of the others' states (225 each way), 2 us in
// all, so clusters are for steps of more entries than one CTA takes in a pass
// or two (bucket_group_us in plan.cu).  Measured, one CTA / eight, six queries
// one after the other: BiDS on the 2048^2 road graph 108 / 52 ms, ET 228 / 81
// (the queue / bitmap frontier on all CTAs: 105, 96), BiD-A* on 1024^2 11 / 16;
// a 64-leaf star on 2048^2 104 / 25 ms (46 on 32 CTAs of the queue path);
// 256 BiD-A* queries with 64-bit distances on 4096^2, clusters of two: 136 ->
// 106 ms, because the longest queries outlast the rest.
__device__ __forceinline__ void bk_publish(BkShared& sm, u32 par, bool fresh) {
    const u32 t = threadIdx.x;
    BkPub& p = sm.pub[par];
    p.rn[t] = sm.rn[t];
    p.rn[t + 32] = sm.rn[t + 32];
    if (t == 0) {
        p.far_n = sm.far_n;
        p.far_min = sm.far_min;
        p.full = sm.far_n > sm.dev.qcap / 2 && sm.far_n > 2 * sm.far_after;
        p.bound = sm.bound;
        p.late = sm.late;
        p.spill = sm.spill;
        p.fresh = fresh;
        p.cnt0 = sm.cnt_dir[0];
        p.cnt1 = sm.cnt_dir[1];
    }
}

// The state a decision is made from: one CTA's, or all of a cluster's.
struct BkState {
    u32 n0, n1;           // entries of buckets cur + 1 + lane and cur + 33 + lane
    u64 bound, far_min;
    u32 late, spill, farn, full, dry;
};

__device__ __forceinline__ u64 bk_min64(u64 x) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        const u64 y = __shfl_xor_sync(0xffffffffu, x, o);
        x = y < x ? y : x;
    }
    return __shfl_sync(0xffffffffu, x, 0);
}

__device__ __forceinline__ BkState bk_gather(BkShared& sm, u32 cl, u32 par, u32 lo) {
    const u32 t = threadIdx.x;
    cg::cluster_group g = cg::this_cluster();
    BkState s;
    s.n0 = s.n1 = 0;
    for (u32 r = 0; r < cl; ++r) {
        const BkPub* p = g.map_shared_rank(&sm.pub[par], r);
        s.n0 += p->rn[(lo + 1 + t) & (BK_NB - 1)];
        if (t < 31) s.n1 += p->rn[(lo + 33 + t) & (BK_NB - 1)];
    }
    const bool on = t < cl;  // lane r < cl reads CTA r's scalars (cl <= 8: reduced over 8 lanes)
    const BkPub* p = g.map_shared_rank(&sm.pub[par], on ? t : 0u);
    const u32 far = on ? p->far_n : 0u;
    s.bound = bk_min64(on ? p->bound : INF64);
    s.far_min = bk_min64(far ? p->far_min : INF64);
    s.farn = __reduce_add_sync(0xffffffffu, far ? 1u : 0u);
    s.late = __reduce_max_sync(0xffffffffu, on ? p->late : 0u);
    s.spill = __reduce_or_sync(0xffffffffu, on ? p->spill : 0u);
    s.full = __reduce_or_sync(0xffffffffu, on ? p->full : 0u);
    const u32 c0 = __reduce_add_sync(0xffffffffu, on ? p->cnt0 : 0u);
    const u32 c1 = __reduce_add_sync(0xffffffffu, on ? p->cnt1 : 0u);
    s.dry = __all_sync(0xffffffffu, !on || p->fresh) && (c0 == 0 || c1 == 0);
    return s;
}

// The next step, decided by the first warp (every lane computes the same).
// fresh: the entry counts per direction are up to date.
template <typename D, int KIND, bool CL>
__device__ __forceinline__ void bk_decide(const EngineArgs& a, const BkCtx<D>& c, BkShared& sm, bool fresh, u32 par) {
    const u32 t = threadIdx.x;
    const u64 cur = sm.cur, curkey = sm.curkey, step = sm.step;
    const i64 koff = sm.key_off;
    const u32 lo = (u32)cur;
    BkState st;
    if (CL) {
        st = bk_gather(sm, c.cl, par, lo);
    } else {
        st.n0 = sm.rn[(lo + 1 + t) & (BK_NB - 1)];
        st.n1 = t < 31 ? sm.rn[(lo + 33 + t) & (BK_NB - 1)] : 0u;
        st.bound = sm.bound;
        st.far_min = sm.far_min;
        st.late = sm.late;
        st.spill = sm.spill;
        st.farn = sm.far_n;
        st.full = st.farn > sm.dev.qcap / 2 && st.farn > 2 * sm.far_after;
        st.dry = fresh && (sm.cnt_dir[0] == 0 || sm.cnt_dir[1] == 0);
    }
    const u64 bound = st.bound, fmin = st.far_min;
    const u32 n0 = st.n0, n1 = st.n1, spill = st.spill, late = st.late, farn = st.farn;
    const u32 m0 = __ballot_sync(0xffffffffu, n0 != 0), m1 = __ballot_sync(0xffffffffu, n1 != 0);
    // buckets ahead of the current one: first non-empty one of the ring, and
    // of the far list (FAR: none, or at least that many)
    constexpr u32 FAR = 1u << 30;
    const u32 k = m0 ? (u32)__ffs(m0) : (m1 ? 32u + (u32)__ffs(m1) : FAR);
    const u32 kf = farn ? (fmin - cur < FAR ? (u32)(fmin - cur) : FAR) : FAR;
    const u32 nn = __shfl_sync(0xffffffffu, m0 ? n0 : n1, (k - 1) & 31);
    const u32 kn = min(k, kf);
    // mu certificate: every stored entry has key > (next bucket - 1) * step
    // (or is a late one), and its prune value is its key less its offset; once
    // that reaches the bound every remaining entry would be pruned.  App. B: a
    // pair of which one side ran dry before mu was set is disconnected.
    bool stop;
    if (bound != INF64) {
        i64 ahead = (i64)((u64)(kn - 1) * step) + 1;  // smallest key left, less curkey
        if (kn == 1 && late) ahead = late != 0xFFFFFFFFu ? 1 - (i64)late : -(i64)curkey;
        stop = !spill && bound > 0 && (i64)curkey + ahead - koff >= (i64)bound;
    } else {
        stop = !bk_one(KIND) && st.dry;
    }
    u32 what = 0, ahead = k;
    if (stop) {
        what = 3;
    } else if (spill || k == FAR || (farn && (kf <= k || kf < BK_NB / 2 || st.full))) {
        const bool none = k == FAR && !farn;
        if (spill && (!sm.recov || none)) {
            // recover spilled entries before they fall behind, at most once
            // between two processed buckets
            what = 2;
        } else if (farn && (kf <= k || kf < BK_NB / 2 || st.full)) {
            // far entries due soon, an empty ring, or a far list filling up
            // with stale entries (re-bucketing drops them)
            what = 1;
        } else if (k == FAR) {
            what = spill ? 2 : 3;
        }
    }
    if (CL && what == 0) {
        // the bucket's entries per CTA, and this one's share of them
        u32 x = 0;
        if (t < c.cl)
            x = min(cg::this_cluster().map_shared_rank(&sm.pub[par], t)->rn[(lo + k) & (BK_NB - 1)], c.cap + c.ob);
#pragma unroll
        for (int o = 1; o < (int)BK_CL_MAX; o <<= 1) {
            const u32 y = __shfl_up_sync(0xffffffffu, x, o);
            if (t >= (u32)o) x += y;
        }
        const u32 total = __shfl_sync(0xffffffffu, x, c.cl - 1), share = (total + c.cl - 1) / c.cl;
        if (t < c.cl) sm.pre[t + 1] = x;
        if (t == 0) {
            sm.pre[0] = 0;
            sm.e0 = min(c.rank * share, total);
            sm.n = min(c.rank * share + share, total);
        }
    }
    if (t == 0) {
        if (CL) {
            sm.bound = bound;
            sm.any_spill = spill;
        }
        if (what == 0) {
            if (!CL) sm.n = min(nn, c.cap + c.ob);
            sm.slot = (lo + k) & (BK_NB - 1);
            sm.recov = 0;
            sm.idle = 0;
            sm.late = 0;  // late entries of this bucket's processing
        } else {
            // the window moves up to the far list's first bucket when the
            // ring holds nothing before it
            const u64 to = (what == 1 && (k == FAR || fmin - cur <= k) && fmin > cur + 1) ? fmin - 1 : cur;
            ahead = 0;
            sm.cur = to;
            sm.curkey = curkey + (to - cur) * step;
            if (what == 2) sm.recov = 1;
            // a bounded number of decisions without a processed bucket: only
            // an internal error gets here, never valid input
            if (++sm.idle > 4096) {
                atomicOr(a.err, ERRB_INTERNAL);
                what = 3;
            }
        }
        if (ahead) {
            sm.cur = cur + ahead;
            sm.curkey = curkey + (u64)ahead * step;
        }
        sm.what = what;
    }
}

// Largest tentative distance of an SSSP group's targets (INF64 while one is
// unreached), by one warp: prune bound and stop certificate (Sec. 4.3).
template <typename D>
__device__ __forceinline__ u64 bk_target_max(const EngineArgs& a, const BkCtx<D>& c, const GroupDev& G) {
    u64 m = 0;
    bool all = true;
    for (u32 q = threadIdx.x & 31u; q < G.qcnt; q += 32) {
        const u64 d = ld_dist(c.dist + a.qedges[G.qbeg + q].b);
        all = all && d != DT<D>::INF;
        m = d > m ? d : m;
    }
    all = __all_sync(0xffffffffu, all);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const u64 y = __shfl_xor_sync(0xffffffffu, m, o);
        m = y > m ? y : m;
    }
    return (all && G.qcnt > 0) ? m : INF64;
}

// Add the warp's net entry counts per direction (pairs, while mu is unset:
// they only serve the disconnected exit).
template <typename D, int KIND>
__device__ __forceinline__ void bk_flush_dir(BkCtx<D>& c, BkShared& sm) {
    if (bk_one(KIND)) return;
    const u32 s0 = __reduce_add_sync(0xffffffffu, (u32)c.dc0);
    const u32 s1 = __reduce_add_sync(0xffffffffu, (u32)c.dc1);
    if ((threadIdx.x & 31) == 0) {
        if (s0) atomicAdd(&sm.cnt_dir[0], s0);
        if (s1) atomicAdd(&sm.cnt_dir[1], s1);
    }
    c.dc0 = c.dc1 = 0;
}

// One group, or (BK_MULTI) search `rank` of one.  Returns false when a wait of
// the team ran out.
template <typename D, int B, int KIND, bool CL>
__device__ __forceinline__ bool bk_group(const EngineArgs& a, const TeamCtx& tc, u32 gi, const GroupDev& G,
                                         BkShared& sm, unsigned char* ring) {
    constexpr u32 KS = bk_one(KIND) ? 0u : 1u;
    const u32 t = threadIdx.x, rank = KIND == BK_MULTI || CL ? tc.rank : 0u;
    const u64 t_start = (a.group_ns && t == 0 && rank == 0) ? global_ns() : 0;
    BkCtx<D> c;
    c.dist = reinterpret_cast<D*>(sm.dev.dist);
    c.touched = sm.dev.touched;
    c.tcap = sm.dev.tcap;
    c.cap = a.ring_cap;
    c.ob = sm.dev.ocap / BK_NB;
    c.ring = reinterpret_cast<typename BkEntry<D>::T*>(ring);
    c.mode = G.mode;
    c.target = G.target;
    c.qe = G.qbeg;
    c.ks = KIND == BK_MULTI ? G.kshift : 0u;
    c.i0 = rank;
    c.cl = CL ? tc.size : 1u;
    c.rank = CL ? rank : 0u;
    c.c_x = c.c_e = c.c_r = c.c_p = c.c_t = 0;
    c.dc0 = c.dc1 = 0;
    const u32 flat_range = a.g.n << KS, nwords = (flat_range + 31u) >> 5;
    const u64 step = KIND != BK_SINGLE ? 2 * G.delta : G.delta;
    const u32 scnt = KIND == BK_MULTI ? 1u : G.scnt;  // searches of this CTA
    u32 sdeg = 0;
    const bool lead = !CL || rank == 0;  // a cluster's first CTA starts the searches
    if (t < scnt) {
        const SearchDev s = a.searches[G.sbeg + (KIND == BK_MULTI ? rank : 0u) + t];
        const u32* off = s.dir ? a.g.off_t : a.g.off;
        sdeg = __ldg(off + s.src + 1) - __ldg(off + s.src);
        sm.src[t] = s.src;
        sm.sdir[t] = s.dir;
        sm.pcnt[t] = s.pcnt;
        if (KIND != BK_MULTI && s.pcnt) sm.pcache[t] = a.partners[s.pbeg];
        const u32 f = (s.src << KS) | t;
        if (lead) {
            st_dist(bk_at<D, KIND>(c, f), 0);
            c.touched[t] = f;
        }
        if (t == 0) {
            sm.key_off = KIND == BK_MULTI ? 0 : s.key_off;
            sm.npart = s.pcnt;
            if (a.g.pc != nullptr) {
                sm.pa = a.g.pc[s.src];
                sm.pb = a.g.pc[s.pot_b];
            }
        }
    }
    if (t < BK_NB) sm.rn[t] = 0;
    if (KIND == BK_MULTI && t < KMAX) sm.muj[t] = 0;
    if (t == 0) {
        sm.bound = INF64;
        sm.step = step;
        sm.cur = sm.curkey = 0;
        sm.late = 0;
        sm.far_n = sm.far_at = sm.far_after = 0;
        sm.far_min = INF64;
        sm.tn = lead ? scnt : 0u;
        sm.tov = sm.spill = sm.recov = sm.idle = sm.ndef = 0;
        sm.cnt_dir[0] = sm.cnt_dir[1] = 0;
    }
    if (rank == 0)
        for (u32 q = t; q < G.qcnt; q += B) a.mu[G.qbeg + q] = INF64;
    __syncthreads();
    if (KIND == BK_MULTI) {
        const u32 pbeg = a.searches[G.sbeg + rank].pbeg;
        for (u32 p = t; p < sm.npart; p += B) {
            const PartnerDev pd = a.partners[pbeg + p];
            sm.pj[p] = pd.j;
            sm.qej[pd.j] = pd.qe;
            sm.muj[pd.j] = INF64;
        }
        // every search's source distance and mu are in place
        if (!team_sync(tc, a, &sm.flag)) return false;
    }
    const bool pot = KIND == BK_BIDASTAR || (KIND == BK_SINGLE && c.mode == GM_ASTAR);
    c.d0 = bk_one(KIND) ? sm.sdir[0] : 0u;
    c.dm = bk_one(KIND) ? 0u : sm.sdir[1];
    c.magic = step > 1 ? (u32)((1ull << 32) / step) : 0xFFFFFFFFu;
    c.cur_lo = 0;
    c.kc = sm.key_off;
    // Init: the sources (key 0) go to the first step
    if (lead && t < scnt) bk_insert<D, KIND>(c, sm, (sm.src[t] << KS) | t, sdeg > 4 ? 2u : 0u, -sm.key_off, 0);
    bk_flush_dir<D, KIND>(c, sm);
    __syncthreads();
    u64 rounds = 0;
    bool fresh = false;
    for (u32 par = 0;; par ^= 1u) {
        if (CL) {
            if (t < 32) bk_publish(sm, par, fresh);
            cg::this_cluster().sync();
        }
        if (t < 32) bk_decide<D, KIND, CL>(a, c, sm, fresh, par);
        __syncthreads();
        const u32 what = sm.what;
        if (KIND == BK_MULTI && t == 0) atomicAdd(&tc.ts->progress, 1u);  // the searches that are done wait
        if (what == 3) break;
        c.cur_lo = (u32)sm.cur;
        c.kc = sm.key_off - (i64)sm.curkey;
        fresh = false;
        if (what == 0) {
            bk_process<D, B, KIND, CL>(a, c, sm, pot);
            if (KIND == BK_SINGLE && c.mode == GM_SSSP && lead && t >= B - 32 && (rounds & 3) == 0) {
                __syncwarp();
                const u64 m = bk_target_max<D>(a, c, G);
                if (t == B - 32) atomicMin(reinterpret_cast<unsigned long long*>(&sm.bound), (unsigned long long)m);
            }
            if (KIND == BK_MULTI && t >= B - 32) {
                __syncwarp();
                bk_refresh(a, sm);
            }
            ++rounds;
        } else if (what == 1) {
            bk_redistribute<D, B, KIND>(a, c, sm, pot);
        } else {
            bk_recover<D, B, KIND>(a, c, sm, pot, nwords);
        }
        __syncwarp();
        if (!bk_one(KIND) && what == 0 && (rounds & 15) == 0) {
            // the counts per direction only serve the disconnected exit,
            // which may come some steps later
            bk_flush_dir<D, KIND>(c, sm);
            fresh = true;
        }
        if (what == 0 && t == 0) sm.rn[sm.slot] = 0;  // nothing is inserted into the processed bucket
        __syncthreads();
        if (what == 0 && sm.ndef) {
            bk_deferred<D, B, KIND>(a, c, sm, pot);
            fresh = false;
            __syncthreads();
        }
    }
    // entries left in the spill bitmap by an early stop
    if (CL) cg::this_cluster().sync();  // every CTA has made the last decision, and its writes are done
    if (CL ? sm.any_spill : sm.spill)
        for (u32 w = c.rank * B + t; w < nwords; w += c.cl * B) sm.dev.bm[0][w] = 0u;
    if (KIND == BK_SINGLE && c.mode == GM_SSSP && lead) {
        for (u32 q = t; q < G.qcnt; q += B) {
            const u64 d = ld_dist(c.dist + a.qedges[G.qbeg + q].b);
            a.mu[G.qbeg + q] = (d == DT<D>::INF) ? INF64 : d;
        }
    }
    const u32 tn = min(sm.tn, c.tcap);
    const bool tov = sm.tov != 0;
    if (KIND != BK_MULTI && !CL && a.path_buf != nullptr) {
        __syncthreads();
        TeamCtx one{0, 0, 1, nullptr, false, 1};
        GCtx<D> g;
        g.G = G;
        g.dist = c.dist;
        g.n = a.g.n;
        g.slot = sm.dev;
        find_paths<D, B>(a, one, g, sm, flat_range, tn, tov);
    }
    if (KIND == BK_MULTI) {
        // the other searches read these distances until they end, too
        if (!team_sync(tc, a, &sm.flag)) return false;
    } else if (CL) {
        cg::this_cluster().sync();  // the answers are read
    } else {
        __syncthreads();
    }
    if (tov) {
        for (u32 f = t; f < flat_range; f += B) st_dist(bk_at<D, KIND>(c, f), DT<D>::INF);
    } else {
#pragma unroll 4
        for (u32 k = t; k < tn; k += B) st_dist(bk_at<D, KIND>(c, __ldcg(c.touched + k)), DT<D>::INF);
    }
    if (a.counters) {
        unsigned long long* cp = &a.counters->extracted;
        const u32 mine[5] = {c.c_x, c.c_e, c.c_r, c.c_p, c.c_t};
        const int at[5] = {0, 1, 2, 3, 7};
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            u64 x = mine[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
            if ((t & 31u) == 0 && x) atomicAdd(cp + at[k], (unsigned long long)x);
        }
        if (t == 0 && lead) {
            atomicAdd(cp + 4, (unsigned long long)rounds);
            if (rank == 0) atomicAdd(cp + 5, 1ull);
            atomicAdd(cp + 6, (unsigned long long)scnt);
        }
    }
    if (a.group_ns && t == 0 && rank == 0) a.group_ns[gi] = global_ns() - t_start;
    __syncthreads();
    return true;
}

// Threads per SM the kernel is compiled to keep resident (64 registers).
template <int B>
struct BucketMinBlocks {
    static constexpr int value = 1024 / B;
};

// BK_CTAS: each CTA is a team that takes groups from its queue; no CTA waits
// for another one, so the launch is an ordinary one.  BK_TEAMS: some teams
// have several CTAs and run Multi-BiDS groups, one search per CTA (a
// cooperative launch: the CTAs of a team meet when a group starts and ends).
// BK_CLUSTERS: each cluster of a.cluster CTAs is a team.
template <typename D, int B, int RUN>
__global__ void __launch_bounds__(B, (BucketMinBlocks<B>::value)) bucket_kernel(EngineArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BkShared& sm = *reinterpret_cast<BkShared*>(smem_raw);
    unsigned char* ring = smem_raw + ((sizeof(BkShared) + 15) & ~(size_t)15);
    TeamCtx tc;
    tc.team = RUN == BK_TEAMS ? a.cta_team[blockIdx.x] : RUN == BK_CLUSTERS ? blockIdx.x / a.cluster : a.team0 + blockIdx.x;
    tc.rank = RUN == BK_TEAMS ? blockIdx.x - a.team_first[tc.team] : RUN == BK_CLUSTERS ? blockIdx.x % a.cluster : 0u;
    tc.size = RUN == BK_TEAMS ? a.team_size[tc.team] : RUN == BK_CLUSTERS ? a.cluster : 1u;
    tc.ts = a.tstate + tc.team;
    tc.global_bar = RUN == BK_TEAMS && tc.size > 1;
    tc.expect = tc.size;
    tc.watch = true;
    const u32 qid = a.team_queue[tc.team];
    if (RUN != BK_TEAMS && a.part == 1) cudaTriggerProgrammaticLaunchCompletion();
    if (threadIdx.x == 0) {
        SlotDev s = a.slots[tc.team];
        if (RUN != BK_CTAS && tc.size > 1) {
            // this CTA's share of the slot's lists.  The spill bitmap is
            // shared by a cluster; a search of a team has its own over the
            // vertices, of which both bitmaps together hold one per search
            // (n bits each, rounded up to words, of 2n per search)
            const u32 r = tc.rank, k = tc.size;
            s.ocap = s.ocap / k / BK_NB * BK_NB;
            s.of += (size_t)r * s.ocap;
            s.od = reinterpret_cast<D*>(s.od) + (size_t)r * s.ocap;
            s.qcap /= k;
            s.tcap /= k;
            for (int x = 0; x < 2; ++x) {
                s.q[x] += (size_t)r * s.qcap;
                s.fd[x] = reinterpret_cast<D*>(s.fd[x]) + (size_t)r * s.qcap;
            }
            s.touched += (size_t)r * s.tcap;
            if (RUN == BK_TEAMS) s.bm[0] += (size_t)r * ((a.g.n + 31u) / 32u);
        }
        sm.dev = s;
    }
    if (RUN == BK_CLUSTERS) cg::this_cluster().sync();  // every CTA runs before its shared memory is written
    for (;;) {
        if (threadIdx.x == 0 && tc.rank == 0) {
            const u32 idx = atomicAdd(a.queue_head + qid, 1u);
            const u32 g = idx < a.queue_len[qid] ? a.queue_items[qid][idx] : NONE;
            if (tc.global_bar) tc.ts->group = g;
            if (RUN == BK_CLUSTERS)
                for (u32 r = 0; r < tc.size; ++r) *cg::this_cluster().map_shared_rank(&sm.group, r) = g;
            else
                sm.group = g;
        }
        if (RUN == BK_TEAMS && tc.global_bar) {
            if (!team_sync(tc, a, &sm.flag)) break;
            if (threadIdx.x == 0) sm.group = ld_volatile(&tc.ts->group);
        }
        if (RUN == BK_CLUSTERS)
            cg::this_cluster().sync();
        else
            __syncthreads();
        const u32 gi = sm.group;
        if (gi == NONE) break;
        const GroupDev G = a.groups[gi];
        if (RUN == BK_TEAMS && tc.global_bar) {
            // the team meets when the group starts, when its searches end
            // and (above) before the next one is claimed
            if (tc.rank < G.scnt) {
                if (!bk_group<D, B, BK_MULTI, false>(a, tc, gi, G, sm, ring)) break;
            } else {
                if (!team_sync(tc, a, &sm.flag) || !team_sync(tc, a, &sm.flag)) break;
            }
            if (!team_sync(tc, a, &sm.flag)) break;
            continue;
        }
        constexpr bool CL = RUN == BK_CLUSTERS;
        if (G.mode != GM_BIDIR)
            bk_group<D, B, BK_SINGLE, CL>(a, tc, gi, G, sm, ring);
        else if (a.searches[G.sbeg].pot)
            bk_group<D, B, BK_BIDASTAR, CL>(a, tc, gi, G, sm, ring);
        else
            bk_group<D, B, BK_BIDS, CL>(a, tc, gi, G, sm, ring);
        // the distances are clean, and the group's shared state read by all,
        // before the next one starts
        if (CL) cg::this_cluster().sync();
    }
    // what follows on the stream waits for the second launch only
    if (RUN == BK_CTAS && a.part == 2) cudaGridDependencySynchronize();
}

// ---- host side ----
constexpr size_t BK_SMEM_MAX = 227 * 1024;  // per CTA
static_assert(bucket_smem_bytes<u32>(BK_RING_MAX_32) <= BK_SMEM_MAX && bucket_smem_bytes<u64>(BK_RING_MAX_64) <= BK_SMEM_MAX,
              "the largest rings fit");

template <typename D, int B, int RUN>
static ppsp_status bucket_smem_attr() {
    static std::atomic<bool> done[SMEM_ATTR_DEVICES];
    int dev = 0;
    PPSP_CUDA_TRY(cudaGetDevice(&dev));
    if (dev >= 0 && dev < SMEM_ATTR_DEVICES && done[dev].load(std::memory_order_acquire)) return PPSP_OK;
    PPSP_CUDA_TRY(cudaFuncSetAttribute(bucket_kernel<D, B, RUN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)std::min<size_t>(bucket_smem_bytes<D>(RING_CAP_MAX), BK_SMEM_MAX)));
    if (dev >= 0 && dev < SMEM_ATTR_DEVICES) done[dev].store(true, std::memory_order_release);
    return PPSP_OK;
}

// A launch of `grid` CTAs in clusters of `cluster`.
struct BkClusterLaunch {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    BkClusterLaunch(u32 grid, u32 threads, size_t smem, u32 cluster, cudaStream_t stream) {
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = cluster;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
};

template <typename D, int B, int RUN>
static ppsp_status bucket_launch_t(const EngineArgs& a, u32 grid, cudaStream_t stream) {
    ppsp_status st = bucket_smem_attr<D, B, RUN>();
    if (st != PPSP_OK) return st;
    const size_t smem = bucket_smem_bytes<D>(a.ring_cap);
    if (RUN == BK_TEAMS) {
        EngineArgs args = a;
        void* params[] = {&args};
        PPSP_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)bucket_kernel<D, B, RUN>, dim3(grid), dim3(B), params,
                                                  smem, stream));
    } else if (RUN == BK_CLUSTERS) {
        if (a.cluster < 1 || a.cluster > BK_CL_MAX || grid % a.cluster) return PPSP_ERR_INVALID_ARG;
        BkClusterLaunch l(grid, B, smem, a.cluster, stream);
        PPSP_CUDA_TRY(cudaLaunchKernelEx(&l.cfg, bucket_kernel<D, B, RUN>, a));
    } else if (a.part == 2) {
        // may start once every CTA of the first launch runs, on the SMs left
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(B);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        PPSP_CUDA_TRY(cudaLaunchKernelEx(&cfg, bucket_kernel<D, B, RUN>, a));
    } else {
        bucket_kernel<D, B, RUN><<<grid, B, smem, stream>>>(a);
        PPSP_CUDA_TRY(cudaGetLastError());
    }
    return PPSP_OK;
}

template <typename D, int RUN>
static ppsp_status bucket_launch(const EngineArgs& a, int block_threads, u32 grid, cudaStream_t stream) {
    if (a.ring_cap < 1 || a.ring_cap > RING_CAP_MAX) return PPSP_ERR_INVALID_ARG;
    if (RUN != BK_CLUSTERS && block_threads == 256)
        return bucket_launch_t<D, RUN == BK_CLUSTERS ? 512 : 256, RUN>(a, grid, stream);
    if (block_threads == 512) return bucket_launch_t<D, 512, RUN>(a, grid, stream);
    if (block_threads == 1024) return bucket_launch_t<D, 1024, RUN>(a, grid, stream);
    return PPSP_ERR_INVALID_ARG;
}

// Resident CTAs per SM.
template <typename D, int B, int RUN>
static ppsp_status bucket_occ_t(int* bpsm, u32 ring_cap) {
    ppsp_status st = bucket_smem_attr<D, B, RUN>();
    if (st != PPSP_OK) return st;
    PPSP_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(bpsm, bucket_kernel<D, B, RUN>, B,
                                                                bucket_smem_bytes<D>(ring_cap)));
    return PPSP_OK;
}

template <typename D, int RUN>
static ppsp_status bucket_occ(int block_threads, u32 ring_cap, int* bpsm) {
    if (ring_cap < 1 || ring_cap > RING_CAP_MAX) return PPSP_ERR_INVALID_ARG;
    if (block_threads == 256) return bucket_occ_t<D, 256, RUN>(bpsm, ring_cap);
    if (block_threads == 512) return bucket_occ_t<D, 512, RUN>(bpsm, ring_cap);
    if (block_threads == 1024) return bucket_occ_t<D, 1024, RUN>(bpsm, ring_cap);
    return PPSP_ERR_INVALID_ARG;
}

// Resident clusters of the whole device.
template <typename D, int B>
static ppsp_status bucket_clusters_t(u32 ring_cap, u32 cluster, int* clusters) {
    ppsp_status st = bucket_smem_attr<D, B, BK_CLUSTERS>();
    if (st != PPSP_OK) return st;
    BkClusterLaunch l(cluster, B, bucket_smem_bytes<D>(ring_cap), cluster, 0);
    PPSP_CUDA_TRY(cudaOccupancyMaxActiveClusters(clusters, bucket_kernel<D, B, BK_CLUSTERS>, &l.cfg));
    return PPSP_OK;
}

template <typename D>
static ppsp_status bucket_clusters(int block_threads, u32 ring_cap, u32 cluster, int* clusters) {
    if (ring_cap < 1 || ring_cap > RING_CAP_MAX || cluster < 1 || cluster > BK_CL_MAX) return PPSP_ERR_INVALID_ARG;
    if (block_threads == 512) return bucket_clusters_t<D, 512>(ring_cap, cluster, clusters);
    if (block_threads == 1024) return bucket_clusters_t<D, 1024>(ring_cap, cluster, clusters);
    return PPSP_ERR_INVALID_ARG;
}

}  // namespace ppsp

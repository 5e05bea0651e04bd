// rw_walk.cu -- the random-walk kernel (journey record of Sec. 3.1 with the
// one-step-exact first step of Sec. 5.2).
//
// Persistent kernel, one warp lane per walk.  A warp claims kWalkChunk walk
// indices at a time from a global cursor; lanes whose walks ended take the next
// indices of the warp's pool, so the warp stays full although walk lengths vary
// by orders of magnitude.  The tables hold each node's transitions in 32-byte
// group sectors of four thresholds with the four successors' words beside
// them, so the next node is known when the group arrives.  A hop to a node of
// degree <= 7 reads its group 0 (and group 1 only when the draw passes group
// 0); a hop to a node of higher degree reads the node's summary (half of the
// last threshold of each group; a dense node-indexed region that stays in L2),
// then the one group that holds the drawn successor, at an address the
// successor word gives without a load (nodes of more than 31 neighbours: a
// group base).
//
// What bounds it, and the shape that follows:
//  - Bulk.  A warp takes new walks and a Philox block only between rounds of
//    four hops, so all its lanes are at the same word of their blocks: one
//    Philox evaluation per lane and four hops (drawn per hop, some lane needed
//    one in nearly every hop, and the whole warp waited for it), and the chain
//    of dependent loads of a new walk once per round at most.  On a 64^3
//    7-point grid (500 walks a row, tables in L2) the launch took 23.4 ms with
//    per-hop draws and refills and takes 15.6 ms (1.16e11 hops/s): L1TEX, one
//    32-byte sector per lane and load, 77 % of peak over the launch, its tail
//    included.
//  - Tables beyond L2 (128^3 27-point: one random group sector of DRAM per
//    hop).  16-byte summaries instead of 32 halve the region that has to stay
//    in L2 beside the groups: 126 -> 118 ms of a 5.2e9-hop launch.
//  - The tail.  The launch ends with its longest walk (a row early in the
//    order: 1e4 to 1e5 hops), a chain of dependent reads; drain_walks runs the
//    last walks of a warp with a team of lanes each.  48^3 27-point grid, 20
//    walks a row, longest walk 54,670 hops: 38.7 ms before, 18.3 ms.
//
// Walk w of row k (rows 0..k-1 are homes, ground absorbs):
//   step 1: draw 0 picks an upper neighbour j > k with probability
//           A_kj / sum_{j>k} A_kj (first-step table);
//   step h: draw h-1 picks the next node by the transition thresholds of the
//           current node; ground if the draw is above every threshold;
//   the walk ends at a node < k (home) or at ground; each visit to k counts a
//   return.  Draw s is word (s mod 4) of Philox(s/4, w, k, tag).
// Output: one record per walk, {end node (-1 ground, -2 step cap), returns or
// length}.
#include "rw_internal.h"

namespace rw {

struct WalkParams {
    const MatWalk* __restrict__ mats;   // per matrix: tables, key, tag
    const int32_t* __restrict__ wmat;   // matrix of each walk row (batched launches)
    const int4* __restrict__ wrow;
    const int64_t* __restrict__ wbase;
    const uint32_t* __restrict__ wofs;  // first walk index of each walk row (NULL: 0)
    const int32_t* __restrict__ chunk_row;
    int64_t total;
    unsigned long long* cursor;
    int2* rec;
    unsigned long long* hops;
    DevStatus* st;
    uint64_t max_steps;
    int record_lengths;                 // see WalkLaunch
    int cache_hint;                     // tables larger than the L2: evict_last / evict_first policies
    int huge;                           // some node has more than eight groups
    MatWalk m0;                         // the matrix of a single-matrix launch
};

// Number of thresholds t <= u among the 8 words of a block (padding words are
// 0xFFFFFFFF and are only counted for u = 0xFFFFFFFF, which the callers clamp).
__device__ __forceinline__ uint32_t count_le8(const uint4 a, const uint4 b, uint32_t u) {
    return (uint32_t)(a.x <= u) + (uint32_t)(a.y <= u) + (uint32_t)(a.z <= u) +
           (uint32_t)(a.w <= u) + (uint32_t)(b.x <= u) + (uint32_t)(b.y <= u) +
           (uint32_t)(b.z <= u) + (uint32_t)(b.w <= u);
}

__device__ __forceinline__ uint4 ld_nc4(const uint32_t* p) {
    return __ldg(reinterpret_cast<const uint4*>(p));
}

// A walk past kSpecHops hops prefetches its node's groups to L2 together with
// the summary read: it then waits for one DRAM round trip instead of an L2
// read followed by a DRAM read.  The long walks set the launch's length; for
// the others the extra sectors would cost more than they save.
constexpr uint64_t kSpecHops = 16384u;

// A warp takes new walks, between rounds, once kRefill of its lanes are idle:
// taking them costs a chain of five dependent loads that the whole warp waits
// for.  4, 8, 12 and 16 give 17.9, 18.1, 18.5 and 19.2 ms on the 64^3 7-point
// grid (walks of 16 hops) and 130.9, 130.3, 129.6 and 127.6 ms on the 128^3
// 27-point one (walks of 9).
constexpr int kRefill = 8;

// Once its walks are all started and at most kTeams are left, a warp gives
// each of them kTeamLanes lanes, one per group of its node (see drain_walks).
constexpr int kTeamLanes = 8;
constexpr int kTeams = 32 / kTeamLanes;

// 32 bytes (eight words) in one load with a cache policy; p must be 32-byte aligned (sectors are).
__device__ __forceinline__ void ld_nc8_hint(const uint32_t* p, uint4& lo, uint4& hi, uint64_t pol) {
    asm("ld.global.nc.L2::cache_hint.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8], %9;"
        : "=r"(lo.x), "=r"(lo.y), "=r"(lo.z), "=r"(lo.w), "=r"(hi.x), "=r"(hi.y), "=r"(hi.z), "=r"(hi.w)
        : "l"(p), "l"(pol));
}
// The same where p holds, t and w unchanged elsewhere (no branch).
__device__ __forceinline__ void ld_nc8_if(bool ok, const uint32_t* p, uint4& lo, uint4& hi) {
    asm("{\n\t.reg .pred ok;\n\tsetp.ne.u32 ok, %9, 0;\n\t"
        "@ok ld.global.nc.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t}"
        : "+r"(lo.x), "+r"(lo.y), "+r"(lo.z), "+r"(lo.w), "+r"(hi.x), "+r"(hi.y), "+r"(hi.z), "+r"(hi.w)
        : "l"(p), "r"((uint32_t)ok));
}
__device__ __forceinline__ uint4 ld_nc4_hint(const uint32_t* p, uint64_t pol) {
    uint4 v;
    asm("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
        : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ uint32_t ld_nc_hint(const uint32_t* p, uint64_t pol) {
    uint32_t v;
    asm("ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ void st_rec_hint(int2* p, int2 v, uint64_t pol) {
    asm volatile("st.global.L2::cache_hint.v2.s32 [%0], {%1, %2}, %3;" ::"l"(p), "r"(v.x), "r"(v.y), "l"(pol)
                 : "memory");
}
// Cache policies: keep (evict_last) and stream (evict_first) when `hint`,
// evict_normal for both otherwise.
struct Policies {
    uint64_t keep, stream, normal;
};
__device__ __forceinline__ Policies walk_policies(int hint) {
    Policies p;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p.normal));
    p.keep = p.stream = p.normal;
    if (hint) {
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p.keep));
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p.stream));
    }
    return p;
}

// Word j (0..3) of the four words c.
__device__ __forceinline__ uint32_t pick4(const uint4 c, uint32_t j) {
    return (j & 2u) ? ((j & 1u) ? c.w : c.z) : ((j & 1u) ? c.y : c.x);
}

// Halves of v below h.
__device__ __forceinline__ uint32_t count_lt2(uint32_t v, uint32_t h) {
    return (uint32_t)((v & 0xFFFFu) < h) + (uint32_t)((v >> 16) < h);
}

// Thresholds t <= u among the four words of a group.
__device__ __forceinline__ uint32_t count_le4(const uint4 t, uint32_t u) {
    return (uint32_t)(t.x <= u) + (uint32_t)(t.y <= u) + (uint32_t)(t.z <= u) + (uint32_t)(t.w <= u);
}

// Bulk prefetch of `bytes` (a multiple of 16) at p (16-byte aligned) into L2.
__device__ __forceinline__ void prefetch_l2(const uint32_t* p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes));
}

// One transition from the node of successor word cw with draw u: the least
// slot j whose threshold exceeds u (thresholds do not decrease along the
// slots, the header slot counts as passed), i.e. successor j - 1, ground if
// there is none among the node's deg + 1 slots.  Returns that successor's
// word, kGroundWord when the walk is absorbed.  n: the matrix's node count
// (the summaries start at sector 2n, the fixed group slots at 3n).  spec:
// prefetch the node's groups to L2 before the summary read returns.
__device__ __forceinline__ uint32_t hop_node(const uint32_t* __restrict__ tab, const uint32_t* __restrict__ gbase,
                                             uint32_t n, uint32_t cw, uint32_t u, const Policies& pol, bool spec) {
    const uint32_t node = cw & kNodeMask;
    const uint32_t cls = cw >> 28;
    const bool big = cls > 2u;  // has a summary: that first, then one group; otherwise group 0, then group 1 if passed
    uint32_t g0 = big ? 3u * n + 8u * node : 2u * node;
    uint32_t g = 0u, ng = cls;
    uint4 t, w;
    if (big) {
        if (cls == kHugeClass) {
            g0 = ld_nc_hint(gbase + node, pol.keep);
            ng = (__ldg(tab + (size_t)g0 * 8u + 4u) + 4u) >> 2;
        } else if (spec) {
            prefetch_l2(tab + (size_t)g0 * 8u, cls * 32u);
        }
        const uint4 s = ld_nc4_hint(tab + (size_t)n * 16u + (size_t)node * 4u, pol.keep);
        const uint32_t uh = u >> 16;
        g = count_lt2(s.x, uh) + count_lt2(s.y, uh) + count_lt2(s.z, uh) + count_lt2(s.w, uh);
    }
    // one iteration; another only past a threshold with the draw's upper half
    // (a summary), or when u passes group 0 (no summary)
    for (; g < ng; ++g) {
        ld_nc8_hint(tab + ((size_t)g0 + g) * 8u, t, w, big ? pol.stream : pol.normal);
        const uint32_t c = count_le4(t, u);
        if (c < 4u) return pick4(w, c);
    }
    return kGroundWord;
}

// First step of a walk from the row whose group 0 is sector g0, lower degree
// lo: the successor word of successor lo + m.
__device__ __forceinline__ uint32_t first_successor(const uint32_t* __restrict__ tab, uint32_t g0, uint32_t lo,
                                                    uint32_t m) {
    const uint32_t slot = lo + m + 1u;
    return __ldg(tab + ((size_t)g0 + (slot >> 2)) * 8u + 4u + (slot & 3u));
}

// First step of a walk with draw u: the least m with u < ft_m among the upper
// neighbours of its row (wrow entry info), else the last.
__device__ __forceinline__ uint32_t first_step(const uint32_t* __restrict__ tab, const uint32_t* __restrict__ fthr,
                                               const int4& info, uint32_t u) {
    const uint32_t* fb = fthr + (size_t)info.y * 8u;
    const uint4 a = ld_nc4(fb), b = ld_nc4(fb + 4);
    const uint32_t up = a.x;
    uint32_t m = (uint32_t)(a.z <= u) + (uint32_t)(a.w <= u) + (uint32_t)(b.x <= u) + (uint32_t)(b.y <= u) +
                 (uint32_t)(b.z <= u) + (uint32_t)(b.w <= u);
    if (m == 6u && up > 6u) {
        for (uint32_t blk = 1;; ++blk) {
            const uint4 c = ld_nc4(fb + 8u * blk), d = ld_nc4(fb + 8u * blk + 4u);
            const uint32_t cnt = count_le8(c, d, u);
            m += cnt;
            if (cnt < 8u || m >= up) break;
        }
    }
    return first_successor(tab, (uint32_t)info.z, (uint32_t)info.w, min(m, up - 1u));
}

// One hop of up to kTeams walks held by single lanes: team t (lanes 8t..8t+7)
// reads the groups of the node of lane `owner` (-1: no walk), and the lane
// that is the my_team-th owner gets its successor word.
__device__ __forceinline__ uint32_t hop_teams(const uint32_t* __restrict__ tab, uint32_t n, int owner, int my_team,
                                              uint32_t coff, uint32_t u) {
    const unsigned lane = lane_id(), t0 = lane & ~(unsigned)(kTeamLanes - 1), q = lane & (kTeamLanes - 1);
    const uint32_t cw = __shfl_sync(kFull, coff, max(owner, 0)), ut = __shfl_sync(kFull, u, max(owner, 0));
    const uint32_t ng = owner < 0 ? 0u : cw >> 28, node = cw & kNodeMask;
    const uint32_t sec = (ng > 2u ? 3u * n + 8u * node : 2u * node) + q;
    uint4 t = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu), w = t;
    ld_nc8_if(q < ng, tab + (size_t)sec * 8u, t, w);
    const uint32_t mine = ut < t.x ? w.x : ut < t.y ? w.y : ut < t.z ? w.z : w.w;
    const uint32_t g = __popc((__ballot_sync(kFull, t.w <= ut) >> t0) & ((1u << kTeamLanes) - 1u));
    uint32_t nw = __shfl_sync(kFull, mine, (int)(t0 + (g & (kTeamLanes - 1))));
    if (g >= ng) nw = kGroundWord;
    return __shfl_sync(kFull, nw, (my_team & (kTeams - 1)) * kTeamLanes);
}

// State of one walk.  Every warp runs its walks four hops at a time (one
// Philox block), so between two rounds each walk's h is a multiple of 4 and
// its next draw is word 0 of block h / 4.
struct WalkState {
    int64_t widx;
    uint64_t h;
    uint32_t k, w, coff, ret;
};

__device__ __forceinline__ uint32_t philox_word(const Philox4& r, uint32_t q) {
    return q == 0u ? r.v0 : q == 1u ? r.v1 : q == 2u ? r.v2 : r.v3;
}

// The record of a walk of h hops that ended at `end` (see WalkLaunch).
__device__ __forceinline__ int2 walk_record(int mode, int32_t end, uint64_t h, uint32_t ret) {
    return make_int2(mode == 2 ? (int32_t)(uint32_t)h : end, (int32_t)(mode == 1 ? (uint32_t)h : ret));
}

// Hops of the block that starts at hop h before the step cap is reached (4: all).
__device__ __forceinline__ uint32_t block_room(uint64_t max_steps, uint64_t h) {
    const uint64_t left = max_steps > h ? max_steps - h : 0u;
    return left < 4u ? (uint32_t)left : 4u;
}

// The last walks of a warp (nothing left to start): the launch cannot end
// before its longest walk, a chain of dependent table reads.  Each walk gets a
// team of eight lanes that read all group sectors of its node at once (lane q
// group q), so a hop waits for one memory round trip instead of a summary and
// then a group; the group that holds the successor is the number of groups
// whose last threshold is passed (one ballot).  The code between two loads is
// straight-line; the next block of draws is computed while loads are in
// flight.  Lanes of a team hold the same state.  Runs until every walk has
// ended or one is within a block of the step cap; the walks left are then in
// the teams' first lanes.  48^3 27-point grid, 20 walks a row, longest walk
// 54,670 hops: 38.7 ms with the last walks in single lanes, 18.3 ms with teams.
// Launches with a node of more than eight groups (more than 31 neighbours) keep
// single lanes throughout: a team has a lane for each of eight groups.  The same
// grid, 200 walks a row: 26 ms, and 43 ms with one row of 1000 neighbours more
// (49 ms before the rounds of four hops).
template <bool MULTI>
__device__ __forceinline__ void drain_walks(const WalkParams& P, bool& active, WalkState& S, int32_t& m,
                                            unsigned long long& my_hops, const Policies& pol) {
    const unsigned lane = lane_id();
    const unsigned t0 = lane & ~(unsigned)(kTeamLanes - 1), q = lane & (kTeamLanes - 1);
    const unsigned live = __ballot_sync(kFull, active);
    bool run = (int)(lane / kTeamLanes) < __popc(live);
    const int src = run ? (int)__fns(live, 0, (int)(lane / kTeamLanes) + 1) : 0;
    S.widx = __shfl_sync(kFull, S.widx, src);
    S.h = __shfl_sync(kFull, S.h, src);
    S.k = __shfl_sync(kFull, S.k, src);
    S.w = __shfl_sync(kFull, S.w, src);
    S.coff = __shfl_sync(kFull, S.coff, src);
    if (!run) S.coff = kGroundWord;  // a team without a walk reads nothing (its matrix may have no tables)
    S.ret = __shfl_sync(kFull, S.ret, src);
    const MatWalk* mw = &P.m0;
    if (MULTI) {
        if (my_hops) atomicAdd(P.hops + m, my_hops);
        my_hops = 0;
        m = __shfl_sync(kFull, m, src);
        if (run) mw = P.mats + m;
    }
    const uint32_t* const tab = mw->tab + 8u * q;
    const uint32_t n3 = 3u * mw->n, key0 = mw->key0, key1 = mw->key1, tag = mw->tag;
    Philox4 rnd = philox4x32_10((uint32_t)(S.h >> 2), S.w, S.k, tag, key0, key1);
    uint32_t last = kGroundWord, steps = 0u;  // how the walk ended in this block, after how many of its hops
    auto hop = [&](uint32_t u) {
        const uint32_t ng = S.coff >> 28, node = S.coff & kNodeMask;
        const uint32_t sec = ng > 2u ? n3 + 8u * node : 2u * node;
        uint4 t = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu), w = t;
        ld_nc8_if(q < ng, tab + (size_t)sec * 8u, t, w);
        const uint32_t mine = u < t.x ? w.x : u < t.y ? w.y : u < t.z ? w.z : w.w;
        const uint32_t g = __popc((__ballot_sync(kFull, t.w <= u) >> t0) & ((1u << kTeamLanes) - 1u));
        uint32_t nw = __shfl_sync(kFull, mine, (int)(t0 + (g & (kTeamLanes - 1))));
        if (g >= ng) nw = kGroundWord;
        const uint32_t nb = nw & kNodeMask;
        // an ended walk stays on kGroundWord (class 0: no loads), which is above every k
        steps += run ? 1u : 0u;
        last = run ? nw : last;
        run = run && nw != kGroundWord && nb >= S.k;
        S.ret += (run && nb == S.k) ? 1u : 0u;
        S.coff = run ? nw : kGroundWord;
    };
    for (uint32_t round = 0;; ++round) {
        const bool near_cap = run && S.h + 4u > P.max_steps;
        if (!__any_sync(kFull, run) || __any_sync(kFull, near_cap)) break;
        if ((round & 1023u) == 0u && __any_sync(kFull, ld_relaxed_u32(&P.st->walk_cap) != 0u)) {
            // another walk hit the step cap: stop (the build reports the error), all lanes together: the
            // loads of the lanes need not see one value, and the rounds' shuffles take the whole warp
            if (run && q == 0u) P.rec[S.widx] = walk_record(P.record_lengths, -2, S.h, S.ret);
            run = false;
            break;
        }
        const Philox4 r = rnd;
        const bool was = run;
        steps = 0u;
        hop(r.v0);
        rnd = philox4x32_10((uint32_t)(S.h >> 2) + 1u, S.w, S.k, tag, key0, key1);
        hop(r.v1);
        hop(r.v2);
        hop(r.v3);
        if (was && !run && q == 0u) {
            const uint64_t h = S.h + steps;
            P.rec[S.widx] =
                walk_record(P.record_lengths, last == kGroundWord ? -1 : (int32_t)(last & kNodeMask), h, S.ret);
            my_hops += h;
        }
        S.h += 4u;
    }
    active = run && q == 0u;
}

// Five blocks per SM (48 registers) for one matrix: 15.6 ms against 16.4 with
// four on the 64^3 7-point grid, 117 against 116 on the 128^3 27-point one;
// four for several matrices, whose table pointers are per lane (five spill).
template <bool MULTI>
__global__ void __launch_bounds__(256, MULTI ? 4 : 5) k_walk(const WalkParams P) {
    const unsigned lane = lane_id();
    const unsigned lt = lanemask_lt();

    int64_t pool_next = 0, pool_end = 0;
    int32_t pool_row = 0;
    bool exhausted = false;

    bool active = false;
    WalkState S{};
    // the walking lane's matrix (fixed for a single-matrix launch)
    const uint32_t* tab = P.m0.tab;
    const uint32_t* gbase = P.m0.gbase;
    uint32_t key0 = P.m0.key0, key1 = P.m0.key1, tag = P.m0.tag, nn = P.m0.n;
    unsigned long long my_hops = 0;
    int32_t my_m = 0;  // matrix whose hops my_hops holds
    const Policies pol = walk_policies(P.cache_hint);

    for (;;) {
        const unsigned live = __ballot_sync(kFull, active);
        if (exhausted) {
            if (live == 0u) break;
            if (__popc(live) <= kTeams && !P.huge && !__any_sync(kFull, active && S.h + 4u > P.max_steps)) {
                drain_walks<MULTI>(P, active, S, my_m, my_hops, pol);
                if (MULTI && active) {
                    const MatWalk& mw = P.mats[my_m];
                    tab = mw.tab;
                    gbase = mw.gbase;
                    key0 = mw.key0;
                    key1 = mw.key1;
                    tag = mw.tag;
                    nn = mw.n;
                }
                continue;
            }
        }
        // ---- new walks for the idle lanes, from the warp's pool of walk indices ----
        bool fresh = false;
        int4 info = make_int4(0, 0, 0, 0);
        const uint32_t* fthr = P.m0.fthr;
        unsigned idle = 32 - __popc(live) >= kRefill ? ~live : 0u;
        while (idle != 0u && !exhausted) {
            if (pool_next >= pool_end) {
                unsigned long long base = 0;
                if (lane == 0)
                    base = ld_relaxed_u32(&P.st->walk_cap) != 0u
                               ? (unsigned long long)P.total
                               : atomicAdd(P.cursor, (unsigned long long)kWalkChunk);
                base = __shfl_sync(kFull, base, 0);
                if ((int64_t)base >= P.total) {
                    exhausted = true;
                    break;
                }
                pool_next = (int64_t)base;
                pool_end = min((int64_t)base + kWalkChunk, P.total);
                pool_row = P.chunk_row[base / kWalkChunk];
            }
            const int avail = (int)(pool_end - pool_next);
            const int rank = __popc(idle & lt);
            const bool take = !active && rank < avail;
            int32_t r = pool_row;
            if (take) {
                S.widx = pool_next + rank;
                while (P.wbase[r + 1] <= S.widx) ++r;
                info = P.wrow[r];
                if (MULTI) {
                    const int32_t m = P.wmat[r];
                    if (m != my_m) {
                        if (my_hops) atomicAdd(P.hops + my_m, my_hops);
                        my_hops = 0;
                        my_m = m;
                    }
                    const MatWalk& mw = P.mats[m];
                    tab = mw.tab;
                    gbase = mw.gbase;
                    fthr = mw.fthr;
                    key0 = mw.key0;
                    key1 = mw.key1;
                    tag = mw.tag;
                    nn = mw.n;
                }
                S.k = (uint32_t)info.x;
                S.w = (uint32_t)(S.widx - P.wbase[r]) + (P.wofs ? P.wofs[r] : 0u);
                S.h = 0;
                S.ret = 0;
                active = true;
                fresh = true;
            }
            const int ntake = min(__popc(idle), avail);
            const unsigned tm = __ballot_sync(kFull, take);
            pool_row = __shfl_sync(kFull, r, 31 - __clz(tm));
            pool_next += ntake;
            idle = __ballot_sync(kFull, !active);
        }

        // ---- one block of draws, four hops of every active lane ----
        const Philox4 rnd = philox4x32_10((uint32_t)(S.h >> 2), S.w, S.k, tag, key0, key1);
        const uint32_t room = block_room(P.max_steps, S.h);
        if (fresh) {
            S.coff = first_step(tab, fthr, info, rnd.v0);
        } else if (active && (S.h & 4095u) == 0u && ld_relaxed_u32(&P.st->walk_cap) != 0u) {
            // another walk hit the step cap: stop (the build reports the error)
            P.rec[S.widx] = walk_record(P.record_lengths, -2, S.h, S.ret);
            my_hops += S.h;
            active = false;
        }
        const bool spec = S.h >= kSpecHops;
#pragma unroll
        for (uint32_t slot = 0; slot < 4u; ++slot) {
            if (!active || (slot == 0u && fresh)) continue;
            if (slot >= room) {  // the step cap
                atomicAdd(&P.st->walk_cap, 1u);
                P.rec[S.widx] = walk_record(P.record_lengths, -2, P.max_steps, S.ret);
                my_hops += P.max_steps;
                active = false;
                continue;
            }
            const uint32_t nw = hop_node(tab, gbase, nn, S.coff, philox_word(rnd, slot), pol, spec);
            const uint32_t nb = nw & kNodeMask;
            if (nw == kGroundWord || nb < S.k) {  // absorbed, or home
                const uint64_t h = S.h + slot + 1u;
                st_rec_hint(P.rec + S.widx,
                            walk_record(P.record_lengths, nw == kGroundWord ? -1 : (int32_t)nb, h, S.ret),
                            pol.stream);
                my_hops += h;
                active = false;
            } else {
                S.ret += (nb == S.k) ? 1u : 0u;
                S.coff = nw;
            }
        }
        S.h += 4u;
    }
    if (MULTI) {
        if (my_hops) atomicAdd(P.hops + my_m, my_hops);
    } else {
        my_hops = warp_sum(my_hops);
        if (lane == 0 && my_hops) atomicAdd(P.hops, my_hops);
    }
}

rw_status run_walks(rw_context* ctx, const WalkBatch& wb, const WalkLaunch& wl, int2* rec,
                    unsigned long long* d_hops, Pool& pool, float* ms) {
    NvtxRange nvtx_range("rw_walk");
    cudaStream_t s = ctx->stream;
    unsigned long long* cursor = alloc_n<unsigned long long>(pool, 1);
    if (!cursor) return RW_ERR_ALLOC;
    rw_status rc;
    if ((rc = check_cuda(cudaMemsetAsync(cursor, 0, sizeof(unsigned long long), s), "memset")))
        return rc;
    if ((rc = check_cuda(cudaMemsetAsync(d_hops, 0, sizeof(unsigned long long) * wb.nmat, s),
                         "memset")))
        return rc;
    if (wb.total == 0) {
        if (ms) *ms = 0.f;
        return RW_OK;
    }
    const bool multi = wb.nmat > 1;
    WalkParams P{};
    P.mats = wb.mats;
    P.wmat = wb.wmat;
    P.wrow = wb.wrow;
    P.wbase = wb.wbase;
    P.wofs = wb.wofs;
    P.chunk_row = wb.chunk_row;
    P.total = wb.total;
    P.cursor = cursor;
    P.rec = rec;
    P.hops = d_hops;
    P.st = ctx->d_status;
    P.max_steps = wl.max_steps;
    P.record_lengths = wl.record_lengths;
    P.cache_hint = wb.table_bytes * 4u > (uint64_t)ctx->l2_bytes * 3u ? 1 : 0;
    P.huge = wb.huge ? 1 : 0;
    P.m0 = wb.m0;
    int per_sm = ctx->opt.walk_blocks_per_sm;
    if (per_sm <= 0) {
        if ((rc = check_cuda(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                 &per_sm, multi ? k_walk<true> : k_walk<false>, 256, 0),
                             "occupancy")))
            return rc;
        if (per_sm < 1) per_sm = 1;
    }
    int64_t blocks = (int64_t)per_sm * ctx->num_sms;
    const int64_t need = (wb.total + 255) / 256;  // never more lanes than walks
    if (blocks > need) blocks = need;
    if (ms) cudaEventRecord(ctx->ev[0], s);
    RW_COUNT_LAUNCH();
    if (multi) k_walk<true><<<(unsigned)blocks, 256, 0, s>>>(P);
    else k_walk<false><<<(unsigned)blocks, 256, 0, s>>>(P);
    if ((rc = check_launch("walk kernel"))) return rc;
    if (ms) {
        cudaEventRecord(ctx->ev[1], s);
        cudaEventSynchronize(ctx->ev[1]);
        cudaEventElapsedTime(ms, ctx->ev[0], ctx->ev[1]);
    }
    return RW_OK;
}

// ---------------------------------------------------------------------------
// Walk reuse (Algorithm 2 of Sec. 5.3).  The simulated walk is the one k_walk
// runs; besides its own record it yields the legal sub-walks that start at a
// later node k' > k: k' is the least node of the sub-walk until it ends at a
// node below k' (a home of k') or at ground.  The lane keeps the increasing
// stack of such candidate starts above k (the top in registers, the rest in
// local memory, each with its returns so far); a hop to node e first pops
// every candidate above e -- each popped candidate is a finished sub-walk
// ending at e, counted unless it started at the previous hop (a one-step walk,
// whose contribution the first-step rule of Sec. 5.2 makes exact) -- then
// pushes e if it is above the new top, or counts a return if it equals it.
// Sub-walks of one start row never overlap (a start is popped before the same
// node can be pushed again), as the paper requires.  Finished sub-walks go to
// the warp's shared-memory stage and from there, in bulk, to the global
// extra-record arrays {start node, end node or -1, returns}.
struct ReuseParams {
    int32_t* xnode;  // start node
    int32_t* xend;   // end node, -1 ground
    uint32_t* xret;
    unsigned long long* xcount;  // records produced (may exceed xcap: then none past xcap is written)
    int64_t xcap;
    unsigned* overflow;          // walks whose stack outgrew CAP
};

constexpr int kReuseStage = 128;

template <int CAP>
__global__ void __launch_bounds__(256) k_walk_reuse(const WalkParams P, const ReuseParams R) {
    __shared__ int32_t s_node[8][kReuseStage];
    __shared__ int32_t s_end[8][kReuseStage];
    __shared__ uint32_t s_ret[8][kReuseStage];
    const unsigned lane = lane_id();
    const unsigned lt = lanemask_lt();
    const unsigned warp = threadIdx.x >> 5;

    int64_t pool_next = 0, pool_end = 0;
    int32_t pool_row = 0;
    bool exhausted = false;

    bool active = false;
    int64_t widx = 0;
    uint32_t k = 0, w = 0, coff = 0, ret = 0;
    const uint32_t* tab = P.m0.tab;
    const uint32_t* gbase = P.m0.gbase;
    const uint32_t key0 = P.m0.key0, key1 = P.m0.key1, tag = P.m0.tag, nn = P.m0.n;
    uint64_t h = 0;
    unsigned long long my_hops = 0;
    const Policies pol = walk_policies(P.cache_hint);

    uint2 stk[CAP];      // candidates below the top: {node, returns}
    int32_t depth = 0;   // candidates above k (the top one in registers)
    uint32_t top = 0, top_ret = 0;
    bool fresh = false;  // the top was pushed by the previous hop
    int stage_n = 0;     // warp-uniform

    auto flush = [&]() {
        __syncwarp();
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(R.xcount, (unsigned long long)stage_n);
        base = __shfl_sync(kFull, base, 0);
        for (int i = (int)lane; i < stage_n; i += 32) {
            const unsigned long long p = base + (unsigned long long)i;
            if (p < (unsigned long long)R.xcap) {
                R.xnode[p] = s_node[warp][i];
                R.xend[p] = s_end[warp][i];
                R.xret[p] = s_ret[warp][i];
            }
        }
        __syncwarp();
        stage_n = 0;
    };

    unsigned owners = 0u;  // live lanes that the teams serve (sparse rounds), and this lane's team's among them
    int owner = 0, my_team = 0;
    for (;;) {
        unsigned live = __ballot_sync(kFull, active);
        if (exhausted && live == 0u) break;
        // ---- new walks for the idle lanes ----
        bool fresh_walk = false;
        int4 info = make_int4(0, 0, 0, 0);
        unsigned idle = 32 - __popc(live) >= kRefill ? ~live : 0u;
        while (idle != 0u && !exhausted) {
            if (pool_next >= pool_end) {
                unsigned long long base = 0;
                if (lane == 0)
                    base = (ld_relaxed_u32(&P.st->walk_cap) | ld_relaxed_u32(R.overflow)) != 0u
                               ? (unsigned long long)P.total
                               : atomicAdd(P.cursor, (unsigned long long)kWalkChunk);
                base = __shfl_sync(kFull, base, 0);
                if ((int64_t)base >= P.total) {
                    exhausted = true;
                    break;
                }
                pool_next = (int64_t)base;
                pool_end = min((int64_t)base + kWalkChunk, P.total);
                pool_row = P.chunk_row[base / kWalkChunk];
            }
            const int avail = (int)(pool_end - pool_next);
            const int rank = __popc(idle & lt);
            const bool take = !active && rank < avail;
            int32_t r = pool_row;
            if (take) {
                widx = pool_next + rank;
                while (P.wbase[r + 1] <= widx) ++r;
                info = P.wrow[r];
                k = (uint32_t)info.x;
                w = (uint32_t)(widx - P.wbase[r]) + (P.wofs ? P.wofs[r] : 0u);
                h = 0;
                ret = 0;
                depth = 0;
                active = true;
                fresh_walk = true;
            }
            const int ntake = min(__popc(idle), avail);
            const unsigned tm = __ballot_sync(kFull, take);
            pool_row = __shfl_sync(kFull, r, 31 - __clz(tm));
            pool_next += ntake;
            idle = __ballot_sync(kFull, !active);
        }

        // ---- one block of draws, four hops of every active lane ----
        const Philox4 rnd = philox4x32_10((uint32_t)(h >> 2), w, k, tag, key0, key1);
        const uint32_t room = block_room(P.max_steps, h);
        if (fresh_walk) {
            coff = first_step(tab, P.m0.fthr, info, rnd.v0);
            depth = 1;  // the first step's upper neighbour starts the stack
            top = coff & kNodeMask;
            top_ret = 0;
            fresh = true;
        }
        const bool stop = active && !fresh_walk && (h & 4095u) == 0u &&
                          (ld_relaxed_u32(&P.st->walk_cap) | ld_relaxed_u32(R.overflow)) != 0u;
        // the last walks of the warp: a team of lanes reads all groups of each one's node at once (as in
        // drain_walks; the walks and their stacks stay in their lanes)
        live = __ballot_sync(kFull, active);
        const bool sparse = exhausted && !P.huge && live != 0u && __popc(live) <= kTeams;
        if (sparse && live != owners) {
            owners = live;
            const int team = (int)lane / kTeamLanes;
            owner = team < __popc(live) ? (int)__fns(live, 0, team + 1) : -1;
            my_team = __popc(live & lt);
        }
        const int hops_now = __any_sync(kFull, stop) ? 0 : 4;
        if (hops_now == 0 && active) {  // another walk hit the step cap or outgrew its stack: stop
            P.rec[widx] = make_int2(-2, (int32_t)ret);
            my_hops += h;
            active = false;
            depth = 0;
        }
#pragma unroll 1
        for (int slot = 0; slot < hops_now; ++slot) {
            // outcome: 0 idle, 1 moved to node `to`, 2 ended at `to` (home, or -1 ground),
            // 3 stopped (step cap or stack overflow)
            int outcome = 0;
            int32_t to = 0;        // the next node (-1: ground)
            uint32_t to_word = 0;  // its successor word
            const bool hop = active && !(slot == 0 && fresh_walk);
            const uint32_t u = philox_word(rnd, (uint32_t)slot);
            if (hop && (uint32_t)slot >= room) {
                outcome = 3;
                atomicAdd(&P.st->walk_cap, 1u);
            }
            if (sparse) to_word = hop_teams(tab, nn, owner, my_team, coff, u);
            if (hop && outcome == 0) {
                if (!sparse) to_word = hop_node(tab, gbase, nn, coff, u, pol, false);
                const uint32_t nb = to_word & kNodeMask;
                if (to_word == kGroundWord) {
                    outcome = 2;
                    to = -1;
                } else {
                    to = (int32_t)nb;
                    outcome = nb < k ? 2 : 1;
                }
            }
            // ---- pop the candidates above `to` (warp-wide, one per round) ----
            bool pop = (outcome == 1 || outcome == 2) && depth > 0 && to < (int32_t)top;
            while (__any_sync(kFull, pop)) {
                const bool emit = pop && !fresh;
                const unsigned em = __ballot_sync(kFull, emit);
                const int cnt = __popc(em);
                if (stage_n + cnt > kReuseStage) flush();
                if (emit) {
                    const int pos = stage_n + __popc(em & lt);
                    s_node[warp][pos] = (int32_t)top;
                    s_end[warp][pos] = to;
                    s_ret[warp][pos] = top_ret;
                }
                stage_n += cnt;
                if (pop) {
                    fresh = false;
                    --depth;
                    if (depth > 0) {
                        const uint2 t = stk[depth - 1];
                        top = t.x;
                        top_ret = t.y;
                    }
                    pop = depth > 0 && to < (int32_t)top;
                }
            }
            if (outcome == 1) {
                if ((uint32_t)to == k) {
                    ++ret;  // every candidate is above k, so the stack is empty here
                    fresh = false;
                } else if (depth > 0 && (uint32_t)to == top) {
                    ++top_ret;
                    fresh = false;
                } else if (depth > CAP) {
                    atomicAdd(R.overflow, 1u);
                    outcome = 3;
                } else {
                    if (depth > 0) stk[depth - 1] = make_uint2(top, top_ret);
                    ++depth;
                    top = (uint32_t)to;
                    top_ret = 0;
                    fresh = true;
                }
                coff = to_word;
            }
            if (outcome >= 2) {
                P.rec[widx] = make_int2(outcome == 3 ? -2 : to, (int32_t)ret);
                my_hops += h + (uint64_t)slot + (outcome == 2 ? 1u : 0u);
                active = false;
                depth = 0;
            }
        }
        h += 4u;
    }
    if (stage_n > 0) flush();
    my_hops = warp_sum(my_hops);
    if (lane == 0 && my_hops) atomicAdd(P.hops, my_hops);
}

// Extra records -> per walk row: counts, then a scatter into row order (the
// order inside a row is immaterial: the merge only sums them).
__global__ void k_extra_count(int64_t cnt, const int32_t* __restrict__ xnode, const uint32_t* __restrict__ wflag,
                              unsigned long long* rows) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(rows + wflag[xnode[i]], 1ull);
}

__global__ void k_extra_scatter(int64_t cnt, const int32_t* __restrict__ xnode, const int32_t* __restrict__ xend,
                                const uint32_t* __restrict__ xret, const uint32_t* __restrict__ wflag,
                                const int64_t* __restrict__ xbase, unsigned long long* fill, int2* xrec) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t r = wflag[xnode[i]];
        const int64_t p = xbase[r] + (int64_t)atomicAdd(fill + r, 1ull);
        const int32_t e = xend[i];
        xrec[p] = make_int2(e >= 0 ? e : -1, (int32_t)xret[i]);
    }
}

template <int CAP>
static rw_status launch_reuse(rw_context* ctx, const WalkParams& P, const ReuseParams& R) {
    int per_sm = ctx->opt.walk_blocks_per_sm;
    rw_status rc;
    if (per_sm <= 0) {
        if ((rc = check_cuda(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_walk_reuse<CAP>, 256, 0),
                             "occupancy")))
            return rc;
        if (per_sm < 1) per_sm = 1;
    }
    int64_t blocks = (int64_t)per_sm * ctx->num_sms;
    const int64_t need = (P.total + 255) / 256;
    if (blocks > need) blocks = need;
    RW_COUNT_LAUNCH();
    k_walk_reuse<CAP><<<(unsigned)blocks, 256, 0, ctx->stream>>>(P, R);
    return check_launch("walk kernel (reuse)");
}

rw_status run_walks_reuse(rw_context* ctx, const WalkBatch& wb, const WalkLaunch& wl, const Tables& T, int2* rec,
                          unsigned long long* d_hops, Pool& pool, Pool& xpool, float* ms, Extras& X) {
    NvtxRange nvtx_range("rw_walk_reuse");
    cudaStream_t s = ctx->stream;
    const int32_t nw = T.n_walk_rows;
    rw_status rc;
    X = Extras{};
    X.xbase = alloc_n<int64_t>(xpool, nw + 1);
    unsigned long long* cursor = alloc_n<unsigned long long>(pool, 1);
    unsigned long long* xcount = alloc_n<unsigned long long>(pool, 1);
    unsigned* overflow = alloc_n<unsigned>(pool, 1);
    if (!X.xbase || !cursor || !xcount || !overflow) return RW_ERR_ALLOC;
    if ((rc = check_cuda(cudaMemsetAsync(X.xbase, 0, sizeof(int64_t) * (size_t)(nw + 1), s), "memset")) ||
        (rc = check_cuda(cudaMemsetAsync(d_hops, 0, sizeof(unsigned long long), s), "memset")))
        return rc;
    if (wb.total == 0) {
        if (ms) *ms = 0.f;
        return RW_OK;
    }
    WalkParams P{};
    P.wrow = wb.wrow;
    P.wbase = wb.wbase;
    P.wofs = wb.wofs;
    P.chunk_row = wb.chunk_row;
    P.total = wb.total;
    P.cursor = cursor;
    P.rec = rec;
    P.hops = d_hops;
    P.st = ctx->d_status;
    P.max_steps = wl.max_steps;
    P.record_lengths = 0;
    P.cache_hint = wb.table_bytes * 4u > (uint64_t)ctx->l2_bytes * 3u ? 1 : 0;
    P.huge = wb.huge ? 1 : 0;
    P.m0 = wb.m0;
    int64_t cap = (int64_t)(ctx->reuse_ratio * (double)wb.total) + (1 << 16);
    int stack = 64;
    unsigned long long* h64 = static_cast<unsigned long long*>(ctx->h_small);
    for (int attempt = 0;; ++attempt) {
        ReuseParams R;
        R.xnode = alloc_n<int32_t>(xpool, cap);
        R.xend = alloc_n<int32_t>(xpool, cap);
        R.xret = alloc_n<uint32_t>(xpool, cap);
        if (!R.xnode || !R.xend || !R.xret) return RW_ERR_ALLOC;
        R.xcount = xcount;
        R.xcap = cap;
        R.overflow = overflow;
        if ((rc = check_cuda(cudaMemsetAsync(cursor, 0, sizeof(unsigned long long), s), "memset")) ||
            (rc = check_cuda(cudaMemsetAsync(d_hops, 0, sizeof(unsigned long long), s), "memset")) ||
            (rc = check_cuda(cudaMemsetAsync(xcount, 0, sizeof(unsigned long long), s), "memset")) ||
            (rc = check_cuda(cudaMemsetAsync(overflow, 0, sizeof(unsigned), s), "memset")))
            return rc;
        if (ms) cudaEventRecord(ctx->ev[0], s);
        rc = stack == 64 ? launch_reuse<64>(ctx, P, R) : launch_reuse<1024>(ctx, P, R);
        if (rc) return rc;
        if (ms) cudaEventRecord(ctx->ev[1], s);
        if ((rc = check_cuda(cudaMemcpyAsync(h64, xcount, 8, cudaMemcpyDeviceToHost, s), "copy")) ||
            (rc = check_cuda(cudaMemcpyAsync(h64 + 1, overflow, 4, cudaMemcpyDeviceToHost, s), "copy")) ||
            (rc = check_cuda(cudaStreamSynchronize(s), "sync")))
            return rc;
        if (ms) cudaEventElapsedTime(ms, ctx->ev[0], ctx->ev[1]);
        const uint64_t produced = h64[0];
        const unsigned over = static_cast<unsigned>(h64[1] & 0xFFFFFFFFull);
        bool again = false;
        if (over) {
            if (stack == 1024) {
                set_error("walk reuse: %u walks have more than 1024 pending sub-walk starts", over);
                return RW_ERR_CAPACITY;
            }
            stack = 1024;
            again = true;
        } else if ((int64_t)produced > cap) {
            cap = (int64_t)produced;
            again = true;
        }
        if (!again) {
            X.count = (int64_t)produced;
            X.xnode = R.xnode;
            X.xend = R.xend;
            X.xret = R.xret;
            const double ratio = 1.125 * (double)produced / (double)wb.total;
            if (ratio > ctx->reuse_ratio) ctx->reuse_ratio = ratio;
            break;
        }
        xpool.release(R.xnode);
        xpool.release(R.xend);
        xpool.release(R.xret);
        if (attempt >= 2) {
            set_error("walk reuse: extra-record capacity did not settle");
            return RW_ERR_CAPACITY;
        }
    }
    // bucket the extra records by walk row
    unsigned long long* rows = alloc_n<unsigned long long>(pool, nw);
    X.xrec = alloc_n<int2>(xpool, X.count);
    if (!rows || !X.xrec) return RW_ERR_ALLOC;
    if ((rc = check_cuda(cudaMemsetAsync(rows, 0, sizeof(unsigned long long) * (size_t)nw, s), "memset")))
        return rc;
    const int g = grid_for(X.count, 256, ctx->num_sms * 16);
    if (X.count > 0) {
        RW_COUNT_LAUNCH();
        k_extra_count<<<g, 256, 0, s>>>(X.count, X.xnode, T.walk_flag, rows);
        if ((rc = check_launch("extra counts"))) return rc;
    }
    if ((rc = check_cuda(scan_i64(reinterpret_cast<const int64_t*>(rows), X.xbase, nw, s, pool), "scan")) ||
        (rc = check_cuda(cudaMemsetAsync(rows, 0, sizeof(unsigned long long) * (size_t)nw, s), "memset")))
        return rc;
    if (X.count > 0) {
        RW_COUNT_LAUNCH();
        k_extra_scatter<<<g, 256, 0, s>>>(X.count, X.xnode, X.xend, X.xret, T.walk_flag, X.xbase, rows, X.xrec);
        if ((rc = check_launch("extra scatter"))) return rc;
    }
    return RW_OK;
}

}  // namespace rw

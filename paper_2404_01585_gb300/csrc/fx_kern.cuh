// Device-side pieces shared by the kernels of the support-evaluation path (kernels.cu) and of
// the map enumerator, overlap graph and exact MIS (enumerate.cu): the resident graph view, the
// warp depth-first search over label slices, block scans, and the device graph with its
// evaluation workspace.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <chrono>
#include <cstdio>
#include <vector>

#include "fx_dev.h"

namespace fx {

#define FULLMASK 0xFFFFFFFFu

struct DevGraphView {
    const VRec *vrec;
    const uint32_t *runs;
    const int32_t *adj;
    const int32_t *lab_vtx;
    int64_t nv;
    int32_t words;  // used-bitmap words per pattern
    const uint32_t *off;  // [lists x nv][nl + 1] slice table (nullable): adjacency position of the
                          // first neighbour with rank label >= l; entry nl is the row's end
    int32_t nl1;          // nl + 1
    const uint4 *edges;   // edge set of an undirected graph (nullable), see EdgeProbe
    uint32_t eb_mask;     // buckets - 1
    int32_t eb_log, eb_bits;  // log2(buckets); bits of a vertex id
    int64_t dstride;  // directed graphs: nv (records of the out, in and mutual lists follow each
                      // other); undirected: 0 (every direction reads the one neighbour list)
};

// A view that has its slice table and, where a pattern has a cycle, its edge set: kernels compiled for
// it leave the other paths out.
struct FastView : DevGraphView {};
__device__ __forceinline__ bool has_slices(const DevGraphView &G) { return G.off != nullptr; }
__device__ __forceinline__ bool has_edges(const DevGraphView &G) { return G.edges != nullptr; }
__device__ __forceinline__ constexpr bool has_slices(const FastView &) { return true; }
__device__ __forceinline__ constexpr bool has_edges(const FastView &) { return true; }

// ------------------------------------------------------------------ warp depth-first search
struct WarpState {
    int32_t t[MAXN];                    // data vertex bound at each level
    uint32_t lo[MAXN], hi[MAXN];        // driver slice of each level
    uint32_t pos[MAXN], base[MAXN], mask[MAXN];
    uint32_t conf[MAXN];                // backjump conflict set of each level (bits of levels)
    uint32_t clo[MAXN][MAXN - 1], chi[MAXN][MAXN - 1];  // further slices (membership tests)
    int32_t nchk[MAXN];                 // further slices | level of the driver slice << 8
    int32_t level;                      // level at suspension
    int32_t floor;                      // lowest level this search may rebind (1: whole root)
    // --- the fields above are the resumable search state (DFS_SAVE_WORDS words)
    unsigned long long need[MAXN];      // neighbour labels each canonical vertex needs
    LevelPlan L;
    int32_t n;
    int32_t pad[1];
    alignas(16) uint4 C[MAXN];          // what a candidate test at each level needs (level_const)
    // slice cache: the slice of level i's candidates in the list of the vertex bound at level b
    // depends on that vertex only (label and list are fixed by the plan), so it is looked up
    // once per vertex bound there; sc_v[i][b] is the vertex it was looked up for (-1: none)
    int32_t sc_v[MAXN][MAXN];
    uint32_t sc_lo[MAXN][MAXN], sc_hi[MAXN][MAXN];
    // slices of level i+1 in the lists of the candidates of level i's current chunk (one per lane)
    uint2 sl[MAXN - 2][32];
    // per-warp totals of the algorithmic work (kept by lane 0, out of the registers)
    unsigned long long acc_scanned, acc_bound, acc_maps, acc_items;
    uint32_t last_steps;  // chunks of the last search
};

__device__ __forceinline__ bool used_bit(const uint32_t *used, int32_t v) {
    return (__ldcg(used + (v >> 5)) >> (v & 31)) & 1u;
}

// The same for a vertex the whole warp asks about: the bit may be set meanwhile, and the lanes have to
// agree on what they saw.
__device__ __forceinline__ bool warp_used(const uint32_t *used, int32_t v) {
    return __any_sync(FULLMASK, used_bit(used, v));
}

// Slice of v's neighbours in list `dir` (DIR_OUT / DIR_IN / DIR_MUT) carrying rank label `lab`
// (empty when absent).  Per lane: lanes may ask for different vertices.  With the slice table this is
// one access; without it (a graph whose table would be too large) the vertex record and a binary
// search of its label runs.
static __device__ __noinline__ uint2 runs_slice(const VRec *rec, const uint32_t *all_runs, uint32_t lab) {
    const uint4 r = __ldg(reinterpret_cast<const uint4 *>(rec));
    const uint32_t *runs = all_runs + r.y;
    const uint32_t nrun = r.w >> 8;
    uint32_t a = 0, b = nrun;
    while (a < b) {
        const uint32_t m = (a + b) >> 1;
        if ((__ldg(runs + m) >> 24) < lab) a = m + 1; else b = m;
    }
    const uint32_t e = __ldg(runs + a);  // the sentinel's label matches none
    if ((e >> 24) != lab) return make_uint2(0u, 0u);
    return make_uint2(r.x + (e & 0xFFFFFFu), r.x + (__ldg(runs + a + 1) & 0xFFFFFFu));
}

template <class View>
__device__ __forceinline__ uint2 lane_slice(const View &G, int32_t v, uint32_t lab, uint32_t dir) {
    const int64_t row = (int64_t)dir * G.dstride + v;
    if (!has_slices(G)) return runs_slice(G.vrec + row, G.runs, lab);
    const uint32_t *o = G.off + row * G.nl1 + lab;
    return make_uint2(__ldg(o), __ldg(o + 1));
}

// The edge set: one membership test is one cache access instead of a search of a hub's slice.
// Buckets of eight 32-bit entries fill a 32-byte sector.  An edge {a, b} (a < b, ids of `eb_bits`
// bits) is mixed by a bijection of its 2 * eb_bits bits (three Feistel rounds), whose low bits
// choose the bucket and whose high bits, plus one, are the entry, so equal entries mean equal edges.
// An entry that finds its bucket full goes to one of the next three, with the distance in its top
// two bits; a bucket with a free place ends the search.  Built on the first evaluation of a pattern
// with a cycle (dev_edge_set).
constexpr int EDGE_WAYS = 8, EDGE_DIST = 4;
constexpr uint32_t EDGE_DIST_SHIFT = 30;

__device__ __forceinline__ void edge_key(const DevGraphView &G, uint32_t v, uint32_t w, uint32_t &bucket,
                                         uint32_t &entry) {
    uint32_t l = min(v, w), r = max(v, w);
    const int b = G.eb_bits, sh = 32 - b;
    r ^= (l * 0x9E3779B1u) >> sh;
    l ^= (r * 0x85EBCA6Bu) >> sh;
    r ^= (l * 0xC2B2AE35u) >> sh;
    const unsigned long long k = (unsigned long long)l << b | r;
    bucket = (uint32_t)k & G.eb_mask;
    entry = (uint32_t)(k >> G.eb_log) + 1u;
}

struct EdgeProbe {
    uint4 x, y;
    uint32_t bucket, entry;
    __device__ __forceinline__ void load(const DevGraphView &G, int32_t v, int32_t w) {
        edge_key(G, (uint32_t)v, (uint32_t)w, bucket, entry);
        x = __ldg(G.edges + 2 * (size_t)bucket);
        y = __ldg(G.edges + 2 * (size_t)bucket + 1);
    }
    __device__ __forceinline__ bool in(uint32_t e) const {
        return x.x == e || x.y == e || x.z == e || x.w == e || y.x == e || y.y == e || y.z == e || y.w == e;
    }
    __device__ __forceinline__ bool test(const DevGraphView &G) {
        if (in(entry)) return true;
        if (in(0u)) return false;
        return further(G.edges, G.eb_mask, bucket, entry);
    }
    // the buckets after a full one (rare, and kept out of the searches' code)
    static __device__ __noinline__ bool further(const uint4 *edges, uint32_t mask, uint32_t bucket, uint32_t entry) {
        EdgeProbe E;
        for (uint32_t d = 1; d < EDGE_DIST; d++) {
            const uint32_t nb = (bucket + d) & mask;
            E.x = __ldg(edges + 2 * (size_t)nb);
            E.y = __ldg(edges + 2 * (size_t)nb + 1);
            if (E.in(entry | d << EDGE_DIST_SHIFT)) return true;
            if (E.in(0u)) return false;
        }
        return false;
    }
};

// Position of the first entry >= c in the sorted slice [lo, hi): an eight-way search.  Seven
// independent probes a round cost one cache latency; halving would cost three for the same narrowing.
static __device__ __noinline__ uint32_t slice_pos(const int32_t *adj, uint32_t lo, uint32_t hi, int32_t c,
                                              uint32_t &probes) {
    uint32_t a = lo, len = hi - lo;
    while (len > 8) {
        const uint32_t q = len >> 3;
        uint32_t k = 0;
#pragma unroll
        for (uint32_t j = 1; j < 8; j++) k += __ldg(adj + a + j * q) < c ? 1u : 0u;
        probes += 7;
        // entries before a + k * q are < c; the one at a + (k + 1) * q (if probed) is not
        a += k * q;
        len = k < 7 ? q : len - 7 * q;
        if (k < 7) len += 1;  // the probed bound itself may be the first entry >= c
    }
    uint32_t k = 0;
#pragma unroll
    for (uint32_t j = 0; j < 8; j++)
        if (j < len) k += __ldg(adj + a + j) < c ? 1u : 0u;
    probes += len;
    return a + k;
}

// Whether the sorted slice [lo, hi) holds c, by the same search on equality.
static __device__ __noinline__ bool contains(const int32_t *adj, uint32_t lo, uint32_t hi, int32_t c,
                                         uint32_t &probes) {
    uint32_t a = lo, len = hi - lo;
    while (len > 8) {
        const uint32_t q = len >> 3;
        uint32_t k = 0;
#pragma unroll
        for (uint32_t j = 1; j < 8; j++) k += __ldg(adj + a + j * q) <= c ? 1u : 0u;
        probes += 7;
        a += k * q;  // if present, c is in [a + k q, a + (k + 1) q)
        len = k < 7 ? q : len - 7 * q;
    }
    bool hit = false;
#pragma unroll
    for (uint32_t j = 0; j < 8; j++)
        if (j < len) hit |= __ldg(adj + a + j) == c;
    probes += len;
    return hit;
}

// Slice of level i's candidates in the list of the vertex bound at level b (warp-uniform, looked up
// once per vertex bound there).
template <class View>
__device__ __forceinline__ uint2 bound_slice(const View &G, WarpState &W, int i, int b,
                                             unsigned long long &bytes) {
    if (W.sc_v[i][b] == W.t[b]) return make_uint2(W.sc_lo[i][b], W.sc_hi[i][b]);
    const uint2 r = lane_slice(G, W.t[b], W.L.lab[i], (W.L.bdir[i] >> (2 * b)) & 3u);
    bytes += 8;
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        W.sc_lo[i][b] = r.x;
        W.sc_hi[i][b] = r.y;
        W.sc_v[i][b] = W.t[b];
    }
    return r;
}

// Constants of a level, one 16-byte read: x, y = the rank labels (< 64) its vertex's neighbours need;
// z = degree | injectivity levels << 8 | backward levels << 16; w = label of the next level | list
// direction there << 8 | 1 << 16 when the next level hangs on this one.  A level's candidates are
// neighbours of the vertices at its backward levels, hence differ from them: only the other levels of
// the same label remain for the injectivity test.
__device__ __forceinline__ uint4 level_const(const LevelPlan &L, int n, int i, unsigned long long need) {
    const uint32_t bm = L.bmask[i];
    const bool ahead = i + 1 < n && (L.bmask[i + 1] >> i & 1u);
    uint4 c;
    c.x = (uint32_t)need;
    c.y = (uint32_t)(need >> 32);
    c.z = L.deg[i] | (uint32_t)(L.injmask[i] & ~bm) << 8 | bm << 16;
    c.w = ahead ? (L.lab[i + 1] | ((uint32_t)(L.bdir[i + 1] >> (2 * i)) & 3u) << 8 | 1u << 16) : 0u;
    return c;
}

// Prepare level i: slices of the bound neighbours at every backward level; the shortest one
// drives the scan (its bounds in dlo, dhi), the others are membership tests.  False if some slice
// is empty.  `pre` is the slice in the list of the vertex bound at level i - 1, when has_pre.
template <class View>
__device__ __forceinline__ bool enter_level(const View &G, WarpState &W, int i,
                                            unsigned long long &bytes, uint32_t &dlo, uint32_t &dhi,
                                            bool has_pre = false, uint2 pre = make_uint2(0u, 0u)) {
    const int lane = threadIdx.x & 31;
    uint32_t bm = W.L.bmask[i], dlen = 0xFFFFFFFFu;
    int nchk = 0, db = 0;
    bool ok = true;
    dlo = dhi = 0;
#pragma unroll 1
    while (bm && ok) {
        const int b = 31 - __clz(bm);  // the newest vertex first: its slice is at hand
        bm &= ~(1u << b);
        const uint2 r = has_pre && b == i - 1 ? pre : bound_slice(G, W, i, b, bytes);
        const uint32_t len = r.y - r.x;
        ok = len != 0;
        const bool shorter = len < dlen;
        if (dlen != 0xFFFFFFFFu) {
            if (lane == 0) {
                W.clo[i][nchk] = shorter ? dlo : r.x;
                W.chi[i][nchk] = shorter ? dhi : r.y;
            }
            nchk++;
        }
        if (shorter) {
            dlo = r.x;
            dhi = r.y;
            dlen = len;
            db = b;
        }
    }
    if (lane == 0) { W.lo[i] = dlo; W.hi[i] = dhi; W.nchk[i] = nchk | db << 8; }
    __syncwarp();
    return ok;
}

// Static one-hop filter: a data vertex can host a pattern vertex only if its degree is at least
// the pattern vertex's and every label the pattern vertex's neighbours carry (ranks < 64) occurs
// among its own neighbours.  Depends on the data vertex alone, so it rejects only vertices that
// belong to no map at all.
__device__ __forceinline__ bool vertex_fits(const DevGraphView &G, int32_t c, uint32_t deg_req,
                                            unsigned long long need) {
    const VRec *r = G.vrec + c;
    const uint32_t deg = __ldg(&r->deg);
    const unsigned long long have = __ldg(reinterpret_cast<const unsigned long long *>(&r->nbr_labels));
    return deg >= deg_req && (have & need) == need;
}

// Dead candidates of a pattern: (level, vertex) pairs found to be in no map that avoids the used set,
// whatever the other levels are bound to -- the search below them failed with a conflict set that
// holds that level alone.  Used sets only grow, so a pair stays dead for the rest of the pattern, for
// every root.  A direct-mapped table of whole keys: a lost entry costs a repeated search, nothing
// else.  In the MiCo-shaped mining run the heaviest six-vertex tree goes from 560 k chunks to 165 k.
constexpr int DEAD_LOG = 12;
__device__ __forceinline__ uint32_t dead_key(int level, int32_t v) { return (uint32_t)(v + 1) | (uint32_t)level << 27; }
__device__ __forceinline__ uint32_t dead_slot(uint32_t key) { return (key * 0x9E3779B1u) >> (32 - DEAD_LOG); }

__device__ __forceinline__ bool level_fits(const DevGraphView &G, int32_t c, const uint4 &C) {
    return vertex_fits(G, c, C.z & 0xFFu, (unsigned long long)C.y << 32 | C.x);
}

// Whether c may be added: not used, fits its pattern vertex, and joined to the vertices t[b] of the
// levels b in `em` (and to `ov`, when >= 0).  With the edge set, all first accesses are issued together;
// one after another they are as many cache latencies.  (Without the set, the callers search the
// slices instead.)
template <class View>
__device__ __forceinline__ bool admit(const View &G, const int32_t *t, const uint4 &C, int32_t c,
                                      const uint32_t *used, uint32_t em, int32_t ov, uint32_t &probes,
                                      const uint32_t *dead = nullptr, int level = 0) {
    const uint32_t uw = used ? __ldcg(used + (c >> 5)) : 0u;
    const uint32_t dk = dead_key(level, c);
    const uint32_t dw = dead ? __ldcg(dead + dead_slot(dk)) : 0u;
    EdgeProbe E;
    const bool probe = ov >= 0 || em;
    if (probe) {
        const int b = __ffs(em) - 1;
        E.load(G, ov >= 0 ? ov : t[b], c);
        if (ov < 0) em &= em - 1;
    }
    const bool fits = level_fits(G, c, C);
    probes += 5;
    if (((uw >> (c & 31)) & 1u) || dw == dk || !fits) return false;
    if (probe && !E.test(G)) return false;
    while (em) {
        const int b = __ffs(em) - 1;
        em &= em - 1;
        E.load(G, t[b], c);
        probes += 8;
        if (!E.test(G)) return false;
    }
    return true;
}

// Candidate test at level i.  rej collects the earlier levels whose bound vertex caused a
// rejection by injectivity (the conflict set of conflict-directed backjumping).
template <class View>
__device__ __forceinline__ bool check_candidate(const View &G, const WarpState &W, const uint4 &C, int i,
                                                int32_t c, const uint32_t *used,
                                                uint32_t &probes, uint32_t &rej, const uint32_t *dead = nullptr) {
    uint32_t im = C.z >> 8 & 0xFFu;
    while (im) {
        const int b = __ffs(im) - 1;
        im &= im - 1;
        if (W.t[b] == c) { rej |= 1u << b; return false; }
    }
    uint32_t bm = C.z >> 16 & 0xFFu;
    int nc = 0;
    if (bm & (bm - 1u)) {
        nc = W.nchk[i];
        bm &= ~(1u << (nc >> 8));
    } else {
        bm = 0;  // one backward level: it drives
    }
    if (!admit(G, W.t, C, c, used, has_edges(G) ? bm : 0u, -1, probes, dead, i)) return false;
    if (!has_edges(G))
        for (int k = 0; k < (nc & 0xFF); k++)
            if (!contains(G.adj, W.clo[i][k], W.chi[i][k], c, probes)) return false;
    return true;
}

// Lexicographically first map (in the level order of W.L) with level 0 bound to `root` and no
// vertex in `used` (nullable).  On success W.t holds the map by level.
//
// Depth-first search with conflict-directed backjumping (Prosser, Computational Intelligence
// 9(3), 1993): when every candidate of level i has failed, the search returns directly to the
// deepest earlier level whose binding could change that outcome -- the levels that define
// level i's candidate slices (its pattern neighbours), the levels whose vertex rejected a
// candidate by injectivity, and the conflict levels handed up by deeper failures.  Levels in
// between cannot make level i succeed, so skipping their remaining candidates removes only
// subtrees without a map: the first map found in lexicographic order is unchanged.
//
// Resumable: when its stop rule says so, the search returns DFS_SUSPENDED before the next
// candidate chunk, with its whole state in W (current level in W.level).  It may later continue
// (resume = true) under a larger used set: bound vertices that have become used are dropped
// (the search continues at the first such level with that level's remaining candidates) and
// every popped candidate is re-tested against the used set.  Everything skipped before the
// suspension failed under the smaller used set and fails under the larger one, so the first map
// found is the first map avoiding the current used set.
enum : int { DFS_NONE = 0, DFS_FOUND = 1, DFS_SUSPENDED = 2, DFS_NOROOM = 3 };

// Counters of the search's algorithmic work (warp-uniform): driver-slice entries scanned, and
// partial maps bound, each weighted by its length (level + 1).
struct SearchWork {
    uint32_t scanned = 0, bound = 0;  // per search: at most budget x 32 entries
};

// Drain: once most warps of a search launch have run out of work items, the searches still
// running suspend at their next check (every DRAIN_EVERY chunks, after DRAIN_MIN_STEPS) instead
// of running to the round's budget, so the launch ends and the next round starts; a suspended
// search resumes (and may be split) there.  Suspension points never change a result.
constexpr uint32_t DRAIN_EVERY = 16;
constexpr uint32_t DRAIN_MIN_STEPS = 32;

__device__ __forceinline__ bool drain_requested(const int32_t *drain) {
    int d = 0;
    if ((threadIdx.x & 31) == 0) d = *reinterpret_cast<const volatile int32_t *>(drain);
    return __shfl_sync(FULLMASK, d, 0) != 0;
}

// When a search stops before it has finished: after `budget` chunks (0: never), or earlier when the
// launch drains.
struct BudgetStop {
    uint32_t budget;
    const int32_t *drain;
    uint32_t next = DRAIN_MIN_STEPS;  // chunks before the next look at `drain`
    __device__ __forceinline__ bool operator()(uint32_t steps) {
        if (!budget) return false;
        if (steps >= budget) return true;
        if (!drain || steps < next) return false;
        next = steps + DRAIN_EVERY;
        return drain_requested(drain);
    }
};

// `stop` is asked, by the whole warp, before every candidate chunk with the chunks scanned so far;
// when it says yes the search is suspended there (DFS_SUSPENDED).
//
// What bounds a search is the chain of dependent cache accesses (most slices are shorter than a
// warp: six entries on average in the MiCo-shaped mining run), so the chain is kept short.  While a
// chunk of level i is tested, every lane also fetches the slice that its candidate gives level
// i + 1; binding a candidate then needs no look-up.  The last level is not entered candidate by
// candidate: all (candidate of level n-2, entry of its slice) pairs of a chunk are tested 32 at a
// time, in lexicographic order (`expand` below).  Together with the slice table and the eight-way
// membership search this took the level-4 candidates of that run from 6.4 M entered levels and as
// many chunks, one after another, to 3.1 M chunks and 1.1 M pair rounds.
// ROOT_KNOWN: the caller has tested the root and passes its level-1 slice.  dead (nullable): the
// pattern's dead candidates, read and added to.
template <class Stop, bool ROOT_KNOWN = false, class View>
__device__ inline int dfs_run(const View &G, WarpState &W, const uint32_t *used, int32_t root,
                              unsigned long long &bytes, uint32_t &probes, uint32_t &steps, bool resume,
                              SearchWork &work, Stop stop, uint2 first = make_uint2(0u, 0u),
                              uint32_t *dead = nullptr) {
    const int lane = threadIdx.x & 31;
    const int n = W.n;
    // the level whose candidates are expanded in pairs: n-2, when the last level hangs on it
    const int xl = n >= 3 && (W.L.bmask[n - 1] >> (n - 2) & 1u) ? n - 2 : -1;
    int i = 1;
    bool ok = true, enter = false;  // enter: level i is to be prepared (one place: the code is large)
    bool has_pre = false;
    uint2 pre = make_uint2(0u, 0u);
    bool fresh = false;    // cc and nx hold the current chunk of level xl
    uint32_t warm = 0;     // levels whose W.sl holds the slices of their current chunk
    int32_t cc = -1;
    uint2 nx = make_uint2(0u, 0u);
    uint32_t hi = 0, pos = 0, base = 0, mask = 0, conf = 0;
    if (!resume) {
        if (lane == 0) { W.t[0] = root; W.floor = 1; }
        __syncwarp();
        if (!ROOT_KNOWN) {
            if (used) {
                bytes += 4;
                if (used_bit(used, root)) return DFS_NONE;
            }
            bytes += 32;
            if (!vertex_fits(G, root, W.L.deg[0], W.need[W.L.vert[0]])) return DFS_NONE;
        }
        pre = first;
        has_pre = ROOT_KNOWN;
        enter = true;
    } else {
        if (used && warp_used(used, W.t[0])) return DFS_NONE;
        i = W.level;
        for (int l = 1; l < i; l++)
            if (used && warp_used(used, W.t[l])) {
                if (l < W.floor) return DFS_NONE;  // a binding this sub-search may not change
                i = l;
                break;
            }
        hi = W.hi[i]; pos = W.pos[i]; base = W.base[i]; mask = W.mask[i]; conf = W.conf[i];
    }
    for (;;) {
        if (enter) {
            uint32_t elo, ehi;
            enter = false;
            conf = 0;
            fresh = false;
            ok = enter_level(G, W, i, bytes, elo, ehi, has_pre, pre);
            if (ok) { hi = ehi; pos = elo; mask = 0; }
        }
        if (!ok) {
            // level i has no candidate left: jump to the deepest level of its conflict set;
            // below the floor the search space of this (sub-)search is exhausted
            const uint32_t cs = (conf | W.L.bmask[i]) & ((1u << i) - 1u);
            const int h = 31 - __clz(cs);
            if (h < W.floor) return DFS_NONE;
            if (dead && cs == 1u << h && lane == 0) {
                const uint32_t k = dead_key(h, W.t[h]);
                dead[dead_slot(k)] = k;
            }
            conf = W.conf[h] | (cs & ~(1u << h));
            i = h;
            hi = W.hi[i]; pos = W.pos[i]; base = W.base[i]; mask = W.mask[i];
            ok = true;
            fresh = false;
            continue;
        }
        if (mask == 0) {
            if (pos >= hi) { ok = false; continue; }
            if (stop(steps)) {
                if (lane == 0) {
                    W.level = i;
                    W.hi[i] = hi; W.pos[i] = pos; W.base[i] = base; W.mask[i] = 0; W.conf[i] = conf;
                }
                __syncwarp();
                return DFS_SUSPENDED;
            }
            const uint32_t k = pos + lane;
            const uint4 C = W.C[i];
            const bool ahead = C.w >> 16;
            bool good = false;
            uint32_t rej = 0;
            if (k < hi) {
                cc = __ldg(G.adj + k);
                if (ahead) nx = lane_slice(G, cc, C.w & 0xFFu, C.w >> 8 & 3u);
                good = check_candidate(G, W, C, i, cc, used, probes, rej, i < n - 1 ? dead : nullptr);
            }
            mask = __ballot_sync(FULLMASK, good);
            if (C.z >> 8 & 0xFFu) conf |= __reduce_or_sync(FULLMASK, rej);
            work.scanned += min(32u, hi - pos);  // slice entries scanned: 4 bytes each in the algorithmic bytes
            steps++;
            base = pos;
            pos += 32;
            fresh = i == xl;
            if (ahead && i != xl) {
                W.sl[i][lane] = nx;
                warm |= 1u << i;
                __syncwarp();
            } else {
                warm &= ~(1u << i);
            }
            continue;
        }
        if (i == xl) {
            // expand: the last level over all candidates of the chunk at once
            const int L = n - 1;
            if (!fresh) {  // resumed, or back from nowhere deeper: fetch the chunk's remaining candidates
                bool live = false;
                if (mask >> lane & 1u) {
                    cc = __ldg(G.adj + base + lane);
                    live = !(used && used_bit(used, cc));
                    nx = lane_slice(G, cc, W.C[i].w & 0xFFu, W.C[i].w >> 8 & 3u);
                }
                mask = __ballot_sync(FULLMASK, live);
                fresh = true;
                if (!mask) continue;
            }
            // the slices that do not depend on the candidate: kept in W.clo/chi[L], the shortest is ks
            const uint4 C = W.C[L];
            const uint32_t lb = (C.z >> 16 & 0xFFu) & ~(1u << i);  // backward levels but this one
            uint32_t bm = lb;
            int nsh = 0, ks = -1, kb = 0;
            uint32_t slo = 0, slen = 0xFFFFFFFFu, empty = 0;
            while (bm) {
                const int b = __ffs(bm) - 1;
                bm &= bm - 1;
                const uint2 r = bound_slice(G, W, L, b, bytes);
                if (r.x == r.y) { empty = 1u << b; break; }
                if (lane == 0) { W.clo[L][nsh] = r.x; W.chi[L][nsh] = r.y; }
                if (r.y - r.x < slen) { slo = r.x; slen = r.y - r.x; ks = nsh; kb = b; }
                nsh++;
            }
            if (lb) __syncwarp();
            if (empty) {  // no candidate of this level can help: only another vertex at that level can
                conf |= empty;
                mask = 0;
                pos = hi;
                continue;
            }
            // each candidate's pairs: the shorter of its own slice and the shortest shared one
            const bool in = mask >> lane & 1u;
            const uint32_t own = in ? nx.y - nx.x : 0u;
            const bool byshare = slen < own;
            const uint32_t len = byshare ? slen : own;
            const uint32_t dlo = byshare ? slo : nx.x;
            uint32_t incl = len;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(FULLMASK, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t excl = incl - len, total = __shfl_sync(FULLMASK, incl, 31);
            const bool anyshare = lb && __any_sync(FULLMASK, byshare && len);
            uint32_t rej = 0;
            uint32_t fm = 0;
            int j = 0;
            int32_t c2 = -1;
            for (uint32_t q0 = 0; q0 < total; q0 += 32) {
                const uint32_t q = q0 + lane;
                j = 0;  // the last lane whose pairs begin at or before q
                for (int o = 16; o > 0; o >>= 1) {
                    const uint32_t e = __shfl_sync(FULLMASK, excl, j + o);
                    if (e <= q) j += o;
                }
                const uint32_t at = __shfl_sync(FULLMASK, dlo, j) + (q - __shfl_sync(FULLMASK, excl, j));
                const int32_t pc = __shfl_sync(FULLMASK, cc, j);
                uint32_t olo = 0, ohi = 0;
                int js = 0;
                if (anyshare) {
                    js = __shfl_sync(FULLMASK, (int)byshare, j);
                    olo = __shfl_sync(FULLMASK, nx.x, j);
                    ohi = __shfl_sync(FULLMASK, nx.y, j);
                }
                bool good = false;
                if (q < total) {
                    c2 = __ldg(G.adj + at);
                    uint32_t im = C.z >> 8 & 0xFFu;
                    good = true;
                    while (im) {
                        const int b = __ffs(im) - 1;
                        im &= im - 1;
                        if ((b == i ? pc : W.t[b]) == c2) {
                            if (b != i) rej |= 1u << b;
                            good = false;
                        }
                    }
                    if (good)
                        good = admit(G, W.t, C, c2, used, has_edges(G) ? (js ? lb & ~(1u << kb) : lb) : 0u,
                                     has_edges(G) && js ? pc : -1, probes);
                    if (!has_edges(G)) {
                        for (int k = 0; good && k < nsh; k++)
                            if (!(js && k == ks)) good = contains(G.adj, W.clo[L][k], W.chi[L][k], c2, probes);
                        if (good && js) good = contains(G.adj, olo, ohi, c2, probes);
                    }
                }
                fm = __ballot_sync(FULLMASK, good);
                steps++;
                work.scanned += min(32u, total - q0);
                if (fm) break;
            }
            if (fm) {
                const int f = __ffs(fm) - 1;
                j = __shfl_sync(FULLMASK, j, f);
                c2 = __shfl_sync(FULLMASK, c2, f);
                const int32_t pc = __shfl_sync(FULLMASK, cc, j);
                // the state is kept at this level from this candidate on, so that a later resume
                // continues past this map (its vertices are used then)
                work.bound += (unsigned)(__popc(mask & ((2u << j) - 1u)) * (i + 1) + n);
                rej = __reduce_or_sync(FULLMASK, rej);
                if (dead && in && lane < j && !(lb | rej)) {
                    const uint32_t k = dead_key(i, cc);
                    dead[dead_slot(k)] = k;
                }
                conf |= rej | lb;
                if (lane == 0) {
                    W.t[i] = pc;
                    W.t[L] = c2;
                    W.level = i;
                    W.hi[i] = hi; W.pos[i] = pos; W.base[i] = base;
                    W.mask[i] = mask & ~((1u << j) - 1u);
                    W.conf[i] = conf;
                }
                __syncwarp();
                return DFS_FOUND;
            }
            work.bound += (unsigned)(__popc(mask) * (i + 1));
            rej = __reduce_or_sync(FULLMASK, rej);
            if (dead && in && !(lb | rej)) {
                const uint32_t k = dead_key(i, cc);
                dead[dead_slot(k)] = k;
            }
            conf |= rej | lb;
            mask = 0;
            continue;
        }
        const int j = __ffs(mask) - 1;
        mask &= mask - 1;
        const int32_t c = __ldg(G.adj + base + j);
        if (resume && used && warp_used(used, c)) continue;  // became used since the chunk scan
        if (lane == 0) W.t[i] = c;
        work.bound += (unsigned)(i + 1);
        if (i == n - 1) {  // keep the position so that a later resume continues past this map
            if (lane == 0) { W.level = i; W.hi[i] = hi; W.pos[i] = pos; W.base[i] = base; W.mask[i] = mask; W.conf[i] = conf; }
            __syncwarp();
            return DFS_FOUND;
        }
        if (lane == 0) { W.pos[i] = pos; W.base[i] = base; W.mask[i] = mask; W.conf[i] = conf; }
        __syncwarp();
        has_pre = warm >> i & 1u;
        if (has_pre) pre = W.sl[i][j];
        ++i;
        enter = true;
    }
}


// Search state of a search that has just found the map in W.t (levels 0 .. n-1), rebuilt from the
// map alone: a following dfs_run with resume goes on past it.  `from` is the first level whose vertex
// may no longer be used.  Nothing is known about why earlier candidates failed, so every level's
// conflict set is all the levels before it (plain backtracking until it is left).
static __device__ __noinline__ void state_of_map(const DevGraphView &G, WarpState &W, int from,
                                             unsigned long long &bytes, uint32_t &probes) {
    const int lane = threadIdx.x & 31;
    const int n = W.n;
    const int xl = n >= 3 && (W.L.bmask[n - 1] >> (n - 2) & 1u) ? n - 2 : -1;
    const int last = xl > 0 && from > xl ? xl : from;
    for (int l = 1; l <= last; l++) {
        uint32_t lo, hi;
        enter_level(G, W, l, bytes, lo, hi);
        const uint32_t at = slice_pos(G.adj, lo, hi, W.t[l], probes);
        __syncwarp();
        if (lane == 0) {
            W.base[l] = at;
            W.pos[l] = at + 1;
            W.mask[l] = l == xl ? 1u : 0u;  // the pairs of the map's own candidate are not finished
            W.conf[l] = (1u << l) - 1u;
            W.level = l;
            W.floor = 1;
        }
        __syncwarp();
    }
}

__device__ __forceinline__ void load_level_plan(WarpState &W, const LevelPlan &L, const Plan &P) {
    const int lane = threadIdx.x & 31;
    constexpr int WORDS = sizeof(LevelPlan) / 4;
    if (lane < WORDS) reinterpret_cast<uint32_t *>(&W.L)[lane] = reinterpret_cast<const uint32_t *>(&L)[lane];
    if (lane < MAXN) {
        W.need[lane] = P.need[lane];
        if (lane < P.n) W.C[lane] = level_const(L, P.n, lane, P.need[L.vert[lane]]);
    }
    if (lane == 0) W.n = P.n;
    // a new plan: no cached slice is valid
    for (int k = lane; k < MAXN * MAXN; k += 32) (&W.sc_v[0][0])[k] = -1;
    __syncwarp();
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULLMASK, v, o);
    return v;
}

// Block-wide exclusive scan of one number per thread; returns the total.
template <class T>
__device__ __forceinline__ T block_scan(T v, T &excl, T *sh /* >= 33 entries */) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(FULLMASK, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        T t = lane < nw ? sh[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const T y = __shfl_up_sync(FULLMASK, t, o);
            if (lane >= o) t += y;
        }
        if (lane < nw) sh[lane] = t;  // inclusive prefix of warp totals
        if (lane == nw - 1) sh[32] = t;
    }
    __syncthreads();
    excl = x - v + (w > 0 ? sh[w - 1] : 0);
    const T total = sh[32];
    __syncthreads();
    return total;
}

#define CK(x)                                                                         \
    do {                                                                              \
        cudaError_t e_ = (x);                                                         \
        if (e_ != cudaSuccess) {                                                      \
            fprintf(stderr, "flexis: %s failed: %s\n", #x, cudaGetErrorString(e_));  \
            return e_ == cudaErrorMemoryAllocation ? FLEXIS_E_NOMEM : FLEXIS_E_CUDA;  \
        }                                                                             \
    } while (0)

struct PatState;
struct Ctl;
struct EnumWS;

// Evaluation workspace: state, plans and results of P patterns; used bitmaps, windows, work items
// and saved searches of H of them (all of them, or none when the streaming greedy evaluates).
struct Workspace {
    int32_t P = 0;           // pattern capacity
    int32_t H = 0;           // patterns with bitmaps, windows and saved searches
    int64_t slots = 0;       // window-slot capacity (H x window size)
    int64_t sel_slots = 0;   // selection-log capacity (patterns x maps)
    int64_t bytes = 0;       // device bytes held
    unsigned char *base = nullptr;  // the allocation that holds the buffers
    PatState *st = nullptr;
    uint32_t *used = nullptr;
    int32_t *dirty = nullptr;
    int32_t clean = 0;  // bitmaps [0, clean) are all zero between evaluations
    int32_t *win_root = nullptr, *win_state = nullptr, *win_map = nullptr;
    int2 *items = nullptr;
    Ctl *ctl = nullptr;
    int32_t *sel_buf = nullptr;
    unsigned long long *mni_seg = nullptr;
    uint32_t *susp = nullptr;
    int32_t *alist = nullptr;
    Plan *plans = nullptr;                   // device plan array (host-plan entry points)
    flexis_support_result *results = nullptr;
    int32_t plans_cap = 0;
    Ctl *h_ctl = nullptr;                    // pinned, and behind it:
    unsigned char *h_stage = nullptr;        // [WS_STAGE] pinned, results on their way to the caller
};

// Buffers of the streaming greedy (stream.cu); all-zero claim words, status words and bitmaps
// between launches (`clean`).
struct StreamWS {
    int32_t S = 0;           // slots
    int64_t ring = 0;        // roots in flight over all slots
    int64_t bytes = 0;
    unsigned char *base = nullptr;  // the allocation that holds the buffers
    bool clean = false;
    size_t zero_bytes = 0;  // from `words` on: claim and status words, bitmaps, dead candidates
    unsigned long long *words = nullptr;
    void *slots = nullptr;
    uint32_t *status = nullptr, *mask = nullptr, *used = nullptr, *dead = nullptr;
    int32_t *maps = nullptr, *dirty = nullptr, *task_links = nullptr;
    uint32_t *tasks = nullptr;
    unsigned char *teams = nullptr;
};

struct DeviceGraph {
    int device = 0;
    cudaStream_t stream = nullptr;
    DevGraphView view{};
    void *d_vrec = nullptr, *d_runs = nullptr, *d_adj = nullptr, *d_labvtx = nullptr, *d_off = nullptr, *d_edges = nullptr;
    bool edges_tried = false;  // dev_edge_set has run
    int64_t n_arcs = 0;
    int64_t bytes = 0;
    int64_t upload_bytes = 0;  // host-to-device bytes of the load (layout arrays, or the edge list)
    int32_t built_on_device = 0;
    int64_t vrec_count = 0, runs_words = 0, adj_words = 0, labvtx_words = 0;  // allocated sizes
    int sm_count = 0, l2 = 0;
    Workspace ws;
    StreamWS sws;
    int stream_per_sm = 0;  // resident blocks of the streaming kernel per SM
    std::atomic<int32_t> servers{0};  // live serving sessions
    int32_t last_P = 0, last_sel = 0;
    cudaEvent_t ev[2]{};
    std::vector<cudaEvent_t> sev;
    cudaGraphExec_t round_exec = nullptr;  // the captured round loop of the last level
    cudaGraphExec_t stream_exec = nullptr; // the captured streaming evaluation,
    std::vector<unsigned char> stream_key; // what it was launched with,
    std::vector<unsigned char> stream_seen; // what the call before was launched with
    int64_t stream_nodes = 0;              // its kernels
    std::vector<cudaEvent_t> gev;          // search-launch events of a group of rounds
    int64_t graph_instantiations = 0, graph_fallbacks = 0;
    int commit_small_blocks = 0;  // one wave of the small-horizon commit kernel
    int32_t max_degree = 0;
    EnumWS *ews = nullptr;        // map enumerator workspace (enumerate.cu), allocated on first use
};

// Map enumerator (enumerate.cu): counts every map of the plans that ask for it into their
// results' n_maps (and materialises maps for the exact MIS); runs on `stream` after the greedy
// phase.  A deadline (measured from t_start) marks unfinished counts FLEXIS_E_TIMEOUT.
int dev_enumerate(DeviceGraph *g, const Plan *d_plans, int32_t P, flexis_support_result *d_results,
                  cudaStream_t stream, const EvalConfig &cfg, flexis_stats *stats,
                  std::chrono::steady_clock::time_point t_start);
void enum_ws_destroy(DeviceGraph *g);

// Exclusive prefix sum of cnt_off[0, n) in place, cnt_off[n] set to the total (enumerate.cu).
// tsum: scratch of scan_tsum_len(n) words.  Three launches on s.
constexpr int SCAN_TILE = 2048;  // elements per block of the scan (1024 threads x 2)
inline long long scan_tsum_len(long long n) { return n / SCAN_TILE + 2; }
int dev_scan_u64(unsigned long long *cnt_off, long long n, unsigned long long *tsum, cudaStream_t s);

// Build the slice table of a resident layout of `nl` rank labels (graph_build.cu); leaves the view
// without one when it would take more than SLICE_TABLE_BYTES or an eighth of the free memory.
constexpr int64_t SLICE_TABLE_BYTES = 4ll << 30;
int dev_slice_table(DeviceGraph *g, int nl);

// Build the edge set of an undirected graph (graph_build.cu), once; leaves the view without one when
// it would take more than EDGE_SET_BYTES or an eighth of the free memory, or an edge finds no place.
constexpr int64_t EDGE_SET_BYTES = 4ll << 30;
int dev_edge_set(DeviceGraph *g);

// The object, stream, events and kernel attributes of a device graph, with no arrays (kernels.cu).
int dev_graph_init(int device, DeviceGraph **out);

}  // namespace fx

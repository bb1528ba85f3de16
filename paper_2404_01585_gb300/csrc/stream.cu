// Streaming greedy: the greedy maximal independent set (Sec. 2.4.3, 3.2.2) of every pattern of a
// batch in one launch, with no batch-wide rounds.
//
// The result is the sequential greedy's: roots in order, each takes its lexicographically first
// map that avoids the vertices of all earlier selections.  Roots are cut into groups of GS
// consecutive ones.  Warps claim groups ahead of the sequential position and search their roots
// against the used set as it is then; groups are retired strictly in order, by one warp at a time:
//   * a root without a map has none under any larger used set: nothing to do;
//   * a map none of whose vertices has been used since is still the root's first map (everything
//     before it in the order was rejected for good): it is selected;
//   * any other map is stale: the retiring warp, which is at the sequential position, searches
//     the root again and gets the sequential greedy's answer.
// Used bits only grow, so a search may read them at any time while they change.
//
// A group's roots are first searched one a lane (lane_searches), then what is left one by one by the
// whole warp.  With as many patterns as warps a warp takes a pattern from its first root to its last.
//
// Who retires: a group's status word has two bits.  DONE is set by the warp that searched it, HEAD
// by the warp that retired the group before it.  Whichever sets the second of the two has the
// role: no warp waits for another, and no group is retired twice.  A slot's claim word holds its
// state (active, done), the warps holding a group of it, the next group and the claim limit, so
// that a claim is one compare-and-swap.  The last warp to let go of a finished pattern writes its
// state, clears what it used and starts the next pattern of the batch in the slot.
//
// How far ahead warps may go adapts per slot.  Stale maps are searched one after another by the
// retiring warp, the rest runs in parallel: an epoch (one window of groups) whose second searches
// took no more chunks than one average group doubles the window, one that took more than four times
// that halves it.  In a model of the MiCo-shaped mining run 5 % of the maps are stale at a
// lag of 32 roots, 20 % at 128, 59 % at 512.
//
// A long search is shared.  When warps are idle, a search of SPLIT_STEPS chunks is cut, as the windowed
// rounds do it, into an ordered list of sub-searches: what it has begun, up to fourteen pieces of the
// unscanned candidates of its shallowest open level, and the rest.  They go to stacks that idle warps
// take from; a task may be cut again.  A task's key is its place in the order (each
// cut divides its key interval by sixteen); the answer is the map found under the smallest key, and
// tasks behind a found one stop.  Nobody waits: the warp that cut the search goes on to other work, and
// the warp that finishes a search's last task takes up the group (or the retiring role) it belongs to.
// The open roots of a group are shared the same way, a task a root.
#include <type_traits>

#include "fx_stream.h"

namespace fx {

namespace {

constexpr int STREAM_WARPS = SEARCH_THREADS / 32;
constexpr unsigned long long W_FIELD = (1ull << 24) - 1;
constexpr int W_NEXT = 24, W_REFS = 48;
static_assert(STREAM_MAX_VERTICES <= (int64_t)W_FIELD * STREAM_GS_MIN, "group numbers");
static_assert(STREAM_MAX_VERTICES < 1ll << 27, "keys of dead candidates");
constexpr unsigned long long W_REF1 = 1ull << W_REFS, W_REFMASK = (1ull << 14) - 1;
constexpr unsigned long long W_ACTIVE = 1ull << 62, W_DONE = 1ull << 63;
enum : uint32_t { G_DONE = 1u, G_HEAD = 2u };
constexpr int G_STEPS = 2;  // above them: chunks scanned in the group
constexpr uint32_t G_STEPS_MAX = (1u << 24) - 1;
enum : int { STOP_NO = 0, STOP_ABORT = 1, STOP_SPLIT = 2 };
constexpr uint32_t STOP_EVERY = 32;     // chunks between looks at the slot's state
constexpr int IDLE_POLLS = 1 << 17;     // looks for work before an idle warp leaves
// Iterations of a lane's search.  (MiCo-shaped mining to 5 edges: 580 ms; 640 when the last three lanes were
// given up after 24 iterations, 600 after 48; 675 with 256 iterations.)
constexpr uint32_t LANE_STEPS = 96;
constexpr uint32_t STREAM_REDO_STEPS = 6;  // set-up of a second search, in chunks
constexpr uint32_t SPLIT_STEPS = 128;   // chunks of a search before it is shared with idle warps
constexpr uint32_t SPLIT_AGAIN = 4096;  // ... before the next try, after one that failed
constexpr int SPLIT_IDLE = 8, SPLIT_READY = 1;  // idle warps, and tasks waiting, that let it be cut
constexpr uint32_t SHARE_STEPS = 128;   // expected chunks of a group's open roots from which they are shared
constexpr int STREAM_BLOCKS = 2;         // resident blocks per SM
constexpr int STREAM_HOME = 16;         // warps that stay with a slot
constexpr unsigned long long SPARE_WAIT = 2000000;  // ns
constexpr int LEAVE_POLLS = 16, LEAVE_POLLS_HOME = 128;  // looks of a roaming and of a home warp in about 1 ms
constexpr uint32_t STREAM_NAP = 1000, STREAM_NAP_HOME = 8000, STREAM_NAP_MAX = 128000;  // ns between looks

// What a retiring warp keeps while one of its searches runs (the kernel has one search call, so that
// the search is inlined with its state in shared memory and the graph's pointers in the parameters).
struct RetireState {
    int64_t count;
    int32_t p, ngroups, rb, re;
    int32_t g, m, redo, pad;
    int32_t lim, window, ep_left, nd;
    uint32_t have, todo;   // roots of the batch with a map; roots not decided yet
    uint32_t whole;        // roots that the whole warp searches (again)
    uint32_t again, got, left;  // roots that lanes search again; with a map then; not decided then
    uint32_t ep_fresh, ep_again;
};

struct StreamWarp {
    WarpState W;
    RetireState R;
    alignas(16) int32_t gm[32][MAXN];  // maps of the roots being retired
};

template <class T>
__device__ __forceinline__ T cg(const T *p) { return __ldcg(p); }

__device__ __forceinline__ unsigned long long word_of(const unsigned long long *w) {
    return *reinterpret_cast<const volatile unsigned long long *>(w);
}

// A search shared by several warps, and what to go on with when it is decided.
struct alignas(16) StreamTeam {
    unsigned long long best;  // smallest (key << 16 | task) of a found map, ~0: none
    int32_t open;             // tasks not finished
    int32_t s, p, g, mode, i;
    uint32_t todo, found, found2, gsteps;
    RetireState R;
    alignas(16) int32_t gm[32][MAXN];
};
static_assert(sizeof(StreamTeam) <= STREAM_TEAM_BYTES, "team record");
// a task: the saved search state, then
constexpr int TASK_TEAM = DFS_SAVE_WORDS, TASK_KEY = DFS_SAVE_WORDS + 1, TASK_SHIFT = DFS_SAVE_WORDS + 3;
static_assert(TASK_SHIFT < STREAM_TASK_WORDS, "task record");
// A cut divides a key interval by 16.  After twelve of them a task that is cut again starts a team of its own:
// where it was left uncut, one task of a six-cycle on 1M vertices ran 190 ms by itself.
constexpr int KEY_BITS = 48, KEY_CUT = 4;
constexpr int TASK_CUT = 1 << KEY_CUT;     // tasks of one block
constexpr int SHIFT_ROOT = 0xFF;           // in TASK_SHIFT: the task is a root of a group, its number the key

__device__ __forceinline__ StreamTeam *team_of(const StreamArgs &A, int t) {
    return reinterpret_cast<StreamTeam *>(A.teams + (size_t)t * STREAM_TEAM_BYTES);
}

// Tasks ready to run: READY_STACKS lock-free stacks.  A cut pushes its tasks, the first on top, with one
// exchange on the stack of its warp; a taker looks at all heads at once and tries the first one that
// is not empty, from a place of its own on.  Last in, first out keeps to the order of the search: the
// tasks of the latest cut, the smallest keys, run first and a map they find stops the others (a queue
// ran twice as many tasks on the 1M-vertex batch).  With a single stack, hundreds of warps cutting and
// thousands taking kept a cut waiting for up to 66 ms.
__device__ int ready_take(const Batch &B, const StreamArgs &A, int start) {  // the whole warp
    const int lane = threadIdx.x & 31;
    int tk = -1;
    for (int b = 0; b < READY_STACKS && tk < 0; b += 32) {
        const int k = (start + b + lane) & (READY_STACKS - 1);
        const unsigned m = __ballot_sync(FULLMASK, (uint32_t)word_of(B.ctl->ready + k) != 0u);
        if (!m) continue;
        const int f = __shfl_sync(FULLMASK, k, __ffs(m) - 1);
        if (lane == 0) {
            unsigned long long *head = B.ctl->ready + f;
            const unsigned long long h = word_of(head);
            if ((uint32_t)h) {
                const int idx = (int)(uint32_t)h - 1;
                const uint32_t nx = (uint32_t)*reinterpret_cast<const volatile int32_t *>(A.task_next + idx);
                if (atomicCAS(head, h, ((h >> 32) + 1) << 32 | nx) == h) {
                    __threadfence();
                    atomicSub(&B.ctl->n_ready, 1);
                    tk = idx;
                }
            }
        }
        tk = __shfl_sync(FULLMASK, tk, 0);
        break;
    }
    return tk;
}

// Tasks t0 .. t0 + n - 1 (the whole warp; their records are written).
__device__ __forceinline__ void ready_put(const Batch &B, const StreamArgs &A, int t0, int n) {
    const int lane = threadIdx.x & 31;
    if (lane < n - 1) A.task_next[t0 + lane] = t0 + lane + 2;  // links hold index + 1
    __threadfence();
    __syncwarp();
    if (lane == 0) {
        unsigned long long *head = B.ctl->ready + ((blockIdx.x * STREAM_WARPS + (threadIdx.x >> 5)) & (READY_STACKS - 1));
        unsigned long long h = word_of(head);
        for (;;) {
            *reinterpret_cast<volatile int32_t *>(A.task_next + t0 + n - 1) = (int32_t)(uint32_t)h;
            __threadfence();
            const unsigned long long prev = atomicCAS(head, h, ((h >> 32) + 1) << 32 | (uint32_t)(t0 + 1));
            if (prev == h) break;
            h = prev;
        }
        atomicAdd(&B.ctl->n_ready, n);
    }
    __syncwarp();
}

// Lock-free stacks of free indices: head = tag << 32 | index + 1; links in next[].  The tag, changed by every
// operation, tells a head apart from an earlier one with the same index.  (One lane.)
__device__ void stack_push(unsigned long long *head, int32_t *next, int idx) {
    unsigned long long h = word_of(head);
    for (;;) {
        *reinterpret_cast<volatile int32_t *>(next + idx) = (int32_t)(uint32_t)h;
        __threadfence();
        const unsigned long long prev = atomicCAS(head, h, ((h >> 32) + 1) << 32 | (uint32_t)(idx + 1));
        if (prev == h) return;
        h = prev;
    }
}

__device__ int stack_pop(unsigned long long *head, const int32_t *next) {
    unsigned long long h = word_of(head);
    while ((uint32_t)h) {
        const int idx = (int)(uint32_t)h - 1;
        const uint32_t nx = (uint32_t)*reinterpret_cast<const volatile int32_t *>(next + idx);
        const unsigned long long prev = atomicCAS(head, h, ((h >> 32) + 1) << 32 | nx);
        if (prev == h) {
            __threadfence();
            return idx;
        }
        h = prev;
    }
    return -1;
}

// An index from a free stack, or a new one below `cap`; -1 when there is none.  (One lane.)
__device__ int take_index(unsigned long long *freed, const int32_t *next, int32_t *bump, int cap) {
    int idx = stack_pop(freed, next);
    if (idx < 0 && *reinterpret_cast<volatile int32_t *>(bump) < cap) {
        idx = atomicAdd(bump, 1);
        if (idx >= cap) idx = -1;
    }
    return idx;
}

// A task of its block is done with.  (One lane.)
__device__ void drop_task(const Batch &B, const StreamArgs &A, int task) {
    const int b = task / TASK_CUT;
    if (atomicSub(A.block_open + b, 1) == 1) stack_push(&B.ctl->blocks_free, A.block_next, b);
}

// Whether the deadline has passed (the whole warp; lane 0 looks).  Warps look between groups, and within a long
// search: most roots are decided in a few steps, so the searches alone would not see the clock.
__device__ __forceinline__ bool late(const Batch &B) {
    if (!B.deadline_ns) return false;
    int r = 0;
    if ((threadIdx.x & 31) == 0 && global_ns() - __ldg(&B.ctl->t0_ns) > B.deadline_ns) {
        *reinterpret_cast<volatile int32_t *>(&B.ctl->expired) = 1;
        r = 1;
    }
    return __shfl_sync(FULLMASK, r, 0) != 0;
}

// Stop rule of a stream search, every STOP_EVERY chunks: abort when the pattern is done, a task ahead
// of this one has found a map, or the deadline has passed; cut the search when it has run for
// `split_at` chunks and warps are idle.
struct StreamStop {
    const unsigned long long *word;
    const unsigned long long *best;  // of the task's team; null: not a task
    unsigned long long key;
    Ctl *ctl;
    unsigned long long deadline_ns;
    uint32_t next, split_at;
    int *reason;  // warp-uniform
    __device__ __forceinline__ bool operator()(uint32_t steps) {
        if (steps < next) return false;
        next = steps + STOP_EVERY;
        int r = STOP_NO;
        if ((threadIdx.x & 31) == 0) {
            if ((word_of(word) & W_DONE) || (best && word_of(best) >> 16 < key)) {
                r = STOP_ABORT;
            } else if (deadline_ns && global_ns() - ctl->t0_ns > deadline_ns) {
                *reinterpret_cast<volatile int32_t *>(&ctl->expired) = 1;
                r = STOP_ABORT;
            } else if (steps >= split_at && *reinterpret_cast<volatile int32_t *>(&ctl->idlers) >= SPLIT_IDLE &&
                       *reinterpret_cast<volatile int32_t *>(&ctl->n_ready) < SPLIT_READY) {  // and take the tasks there are
                r = STOP_SPLIT;
            }
        }
        r = __shfl_sync(FULLMASK, r, 0);
        *reason = r;
        return r != STOP_NO;
    }
};

// Give slot s the next pattern of the batch that has a greedy phase, or leave it empty.  The
// caller is alone on the slot; its bitmap is zero and its group status words are zero.
__device__ __noinline__ void start_slot(const Batch &B, const StreamArgs &A, int s) {
    const int lane = threadIdx.x & 31;
    if (lane == 0) {
        for (;;) {
            const int q = atomicAdd(&B.ctl->next_pattern, 1);
            if (q >= B.P) {
                atomicExch(A.words + s, 0ull);
                break;
            }
            if (B.st[q].phase != PH_GREEDY) {
                atomicAdd(&B.ctl->done_count, 1);
                continue;
            }
            const Plan &P = B.plans[q];
            StreamSlot t;
            t.count = 0;
            t.p = q;
            t.root_begin = P.root_begin;
            t.root_end = P.root_end;
            t.ngroups = (P.root_end - P.root_begin + A.GS - 1) / A.GS;
            t.head = 0;
            t.window = min(A.window0, A.RG);
            t.lim = min(t.ngroups, t.window);
            t.ep_left = t.window;
            t.ep_fresh = t.ep_again = 0;
            t.ndirty = 0;
            t.last_steps = 0;
            A.slots[s] = t;
            A.status[(size_t)s * A.RG] = G_HEAD;
            __threadfence();
            atomicExch(A.words + s, W_ACTIVE | (unsigned long long)t.lim);
            break;
        }
    }
    __syncwarp();
}

__device__ __forceinline__ bool claimable(unsigned long long w) {
    return (w & W_ACTIVE) && !(w & W_DONE) && ((w >> W_NEXT) & W_FIELD) < (w & W_FIELD);
}

// Claim the next group of slot s: its number, or -1.  (Lane 0 works, the warp gets the answer.)
__device__ __forceinline__ int claim(const StreamArgs &A, int s) {
    int g = -1;
    if ((threadIdx.x & 31) == 0) {
        unsigned long long cur = word_of(A.words + s);
        for (int tries = 0; tries < 64 && claimable(cur); tries++) {
            const unsigned long long prev = atomicCAS(A.words + s, cur, cur + (1ull << W_NEXT) + W_REF1);
            if (prev == cur) {
                g = (int)((cur >> W_NEXT) & W_FIELD);
                __threadfence();
                break;
            }
            cur = prev;
        }
    }
    return __shfl_sync(FULLMASK, g, 0);
}

// A slot with a group to claim, looking from slot s0 on; -1 when there is none.
__device__ int find_slot(const StreamArgs &A, int s0) {
    const int lane = threadIdx.x & 31;
    for (int b = 0; b < A.S; b += 32) {
        int s = s0 + b + lane;
        if (s >= A.S) s -= A.S;
        const bool in = b + lane < A.S && s < A.S;
        const bool ok = in && claimable(word_of(A.words + s));
        const unsigned m = __ballot_sync(FULLMASK, ok);
        if (m) return __shfl_sync(FULLMASK, s, __ffs(m) - 1);
    }
    return -1;
}

// Mark the vertices m of the maps of the lanes with `mine` used, listing the words that become
// non-zero; nd counts them (the retiring warp's own copy).
__device__ __noinline__ void use_maps(uint32_t *u, int32_t *dirty, bool mine, const int32_t *m, int n, int &nd) {
    const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
    uint32_t fresh = 0;  // bit l: vertex l opened a word
#pragma unroll
    for (int l = 0; l < MAXN; l++)
        if (mine && l < n && atomicOr(u + ((uint32_t)m[l] >> 5), 1u << (m[l] & 31)) == 0u) fresh |= 1u << l;
    for (int l = 0; l < n; l++) {
        const bool f = fresh >> l & 1u;
        const unsigned b = __ballot_sync(FULLMASK, f);
        const int k = nd + __popc(b & lt);
        if (f && k < DIRTY_CAP) dirty[k] = (int32_t)((uint32_t)m[l] >> 5);
        nd += __popc(b);
    }
}

// The pattern of slot s is finished and no warp holds a group of it: write its state, leave the
// slot clean and start the next pattern in it.
__device__ __noinline__ void end_slot(const Batch &B, const StreamArgs &A, int s, int next) {
    const int lane = threadIdx.x & 31;
    __threadfence();
    const StreamSlot *t = A.slots + s;
    const int p = cg(&t->p), head = cg(&t->head), nd = cg(&t->ndirty);
    if (lane == 0) {
        PatState &S = B.st[p];
        S.rounds = 1;
        S.count = cg(&t->count);
        if (B.sel) S.logged = (int32_t)min(min(S.count, B.plans[p].cap), (int64_t)B.sel_cap);
        S.done = 1;
        S.phase = PH_MNI;
    }
    uint32_t *u = A.used + (size_t)s * B.G.words;
    if (nd <= DIRTY_CAP) {
        for (int k = lane; k < nd; k += 32) u[cg(A.dirty + (size_t)s * DIRTY_CAP + k)] = 0u;
    } else {
        for (int w = lane; w < B.G.words; w += 32) u[w] = 0u;
    }
    uint4 *dead = reinterpret_cast<uint4 *>(A.dead + ((size_t)s << DEAD_LOG));
    for (int k = lane; k < (1 << DEAD_LOG) / 4; k += 32) dead[k] = make_uint4(0u, 0u, 0u, 0u);
    // groups claimed and not retired, and the head's own bit
    const int left = min(max(next - head, 0) + 1, A.RG);
    for (int k = lane; k < left; k += 32) A.status[(size_t)s * A.RG + ((head + k) & (A.RG - 1))] = 0u;
    __threadfence();
    __syncwarp();
    if (lane == 0) atomicAdd(&B.ctl->done_count, 1);
    start_slot(B, A, s);
}

__device__ __forceinline__ void mark_done(const StreamArgs &A, int s) {
    __threadfence();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) atomicOr(A.words + s, W_DONE);
}

// Take the retiring role of slot s at group g.
__device__ __forceinline__ void retire_begin(const StreamArgs &A, StreamWarp &X, int s, int g) {
    const StreamSlot *T = A.slots + s;
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        RetireState &R = X.R;
        R.count = cg(&T->count);
        R.p = cg(&T->p);
        R.ngroups = cg(&T->ngroups);
        R.rb = cg(&T->root_begin);
        R.re = cg(&T->root_end);
        R.lim = cg(&T->lim);
        R.window = cg(&T->window);
        R.ep_left = cg(&T->ep_left);
        R.ep_fresh = cg(&T->ep_fresh);
        R.ep_again = cg(&T->ep_again);
        R.nd = cg(&T->ndirty);
        R.g = g;
        R.m = 0;  // no batch of groups loaded
    }
    __syncwarp();
}

// A lane searches its own root (plain backtracking, one candidate an iteration) while the others search
// theirs: 32 roots for the dependent accesses of one.  Most roots of most patterns are decided within
// a few candidates a level; the ones that are not after LANE_STEPS iterations are left to the whole
// warp (`open`).  Maps go to X.gm; returns the lanes that
// found one.  The per-level positions share W.sl with the warp's searches.
template <class View>
__device__ __forceinline__ uint32_t lane_searches(const View &G, StreamWarp &X, const uint32_t *used,
                                                  uint32_t *dead, bool ok,
                                                  int32_t root, uint2 first, uint32_t &open, uint32_t &iters,
                                                  SearchWork &work) {
    const int lane = threadIdx.x & 31;
    WarpState &W = X.W;
    const int n = W.n;
    int32_t *t = X.gm[lane];
    bool act = ok, found = false;
    int i = 1;
    uint32_t pos = first.x, hi = first.y, tried = 0, bound = 0, probes = 0;
    uint32_t pure = 0;  // levels that hang on the one before alone, with no candidate lost to another level
    __syncwarp();
    if (ok) t[0] = root;
    uint32_t it = 0;
    for (;; it++) {
        if (it >= LANE_STEPS || !__any_sync(FULLMASK, act)) break;
        if (!act) continue;
        if (pos >= hi) {
            // level i is exhausted: when nothing but the vertex at level i - 1 had a part in that, it is
            // dead there; otherwise level i - 1 depends on more than its own slice
            if (i > 1) {
                if (pure >> i & 1u) {
                    const uint32_t k = dead_key(i - 1, t[i - 1]);
                    dead[dead_slot(k)] = k;
                } else {
                    pure &= ~(1u << (i - 1));
                }
            }
            if (--i == 0) {
                act = false;
            } else {
                const uint2 q = W.sl[i - 1][lane];
                pos = q.x;
                hi = q.y;
            }
            continue;
        }
        const int32_t c = __ldg(G.adj + pos);
        pos++;
        tried++;
        const uint4 C = W.C[i];
        uint2 nx = make_uint2(0u, 0u);
        if (C.w >> 16) nx = lane_slice(G, c, C.w & 0xFFu, C.w >> 8 & 3u);
        bool good = true;
        uint32_t im = C.z >> 8 & 0xFFu;
        while (im) {
            const int b = __ffs(im) - 1;
            im &= im - 1;
            good &= t[b] != c;
        }
        if (!good) pure &= ~(1u << i);
        uint32_t bm = C.z >> 16 & 0xFFu;
        if (!(bm & (bm - 1u))) bm = 0;  // one backward level: its slice is what is scanned
        good = good && admit(G, t, C, c, used, has_edges(G) ? bm : 0u, -1, probes, i < n - 1 ? dead : nullptr, i);
        if (!has_edges(G))
            while (good && bm) {
                const int b = __ffs(bm) - 1;
                bm &= bm - 1;
                const uint2 q = lane_slice(G, t[b], W.L.lab[i], (W.L.bdir[i] >> (2 * b)) & 3u);
                good = contains(G.adj, q.x, q.y, c, probes);
            }
        if (!good) continue;
        t[i] = c;
        bound += (unsigned)(i + 1);
        if (i == n - 1) {
            found = true;
            act = false;
            continue;
        }
        W.sl[i - 1][lane] = make_uint2(pos, hi);
        i++;
        // the shortest of the level's slices
        uint32_t nb = W.C[i].z >> 16 & 0xFFu;
        pure = nb == 1u << (i - 1) ? pure | 1u << i : pure & ~(1u << i);
        pos = nx.x;
        hi = nx.y;
        uint32_t len = nb >> (i - 1) & 1u ? hi - pos : 0xFFFFFFFFu;
        nb &= ~(1u << (i - 1));
        while (nb && len) {
            const int b = __ffs(nb) - 1;
            nb &= nb - 1;
            const uint2 q = lane_slice(G, t[b], W.L.lab[i], (W.L.bdir[i] >> (2 * b)) & 3u);
            if (q.y - q.x < len) {
                pos = q.x;
                hi = q.y;
                len = hi - pos;
            }
        }
    }
    iters = it;
    work.scanned += __reduce_add_sync(FULLMASK, tried);
    work.bound += __reduce_add_sync(FULLMASK, bound);
    open = __ballot_sync(FULLMASK, act);
    __syncwarp();
    return __ballot_sync(FULLMASK, found);
}

enum : int { RT_DONE = 0, RT_SEARCH = 1, RT_LANES = 2 };
constexpr int RES_LANES = 100;  // `res`: the lanes have searched X.R.again

// Retire groups, up to 32 roots at a time (a lane per root), until the role passes on or the
// pattern ends (RT_DONE), or roots have to be searched: RT_SEARCH with a root and where to search from,
// or RT_LANES for the roots X.R.again.  `res` >= 0: the outcome of what was asked for last.
//
// Stale maps of a batch are searched again together, a lane a root.  The first of them is at the
// sequential position, so that its new map is final; the others are speculation again.  (One after
// another by the whole warp they took 60 us each, and with the calls in between half of the time of
// the MiCo-shaped run to 5 edges.)
template <class View>
__device__ __forceinline__ int retire_step(const View &G, const Batch &B, const StreamArgs &A, StreamWarp &X, int s, int res,
                                           int32_t &root, int &from) {
    constexpr bool SEL = !std::is_same<View, FastView>::value;  // (selections are logged by the general kernel)
    const int lane = threadIdx.x & 31;
    StreamSlot *T = A.slots + s;
    uint32_t *status = A.status + (size_t)s * A.RG;
    const uint32_t *used = A.used + (size_t)s * B.G.words;
    const int p = X.R.p, ngroups = X.R.ngroups, rb = X.R.rb, re = X.R.re;
    int64_t count = X.R.count;
    int g = X.R.g, m = X.R.m, lim = X.R.lim, window = X.R.window, ep_left = X.R.ep_left, nd = X.R.nd;
    uint32_t have = X.R.have, todo = X.R.todo, whole = X.R.whole, ep_fresh = X.R.ep_fresh, ep_again = X.R.ep_again;
    const Plan &P = B.plans[p];
    const int n = X.W.n;
    const int64_t cap = P.cap;
    const int GS = A.GS, RM = A.RG - 1;
    bool over = false, stopped = false;  // the pattern is finished; the deadline stopped a search
    __syncwarp();
    if (res == RES_LANES) {
        const uint32_t again = X.R.again, got = X.R.got, left = X.R.left;
        have = (have & ~again) | got;
        todo &= ~again | got | left;
        whole |= left;
        ep_again += X.W.last_steps + STREAM_REDO_STEPS;
    } else if (res >= 0) {
        const int redo = X.R.redo;
        ep_again += X.W.last_steps + STREAM_REDO_STEPS;
        if (res == DFS_SUSPENDED) {
            stopped = true;
        } else {
            if (res == DFS_FOUND) {
                if (lane < MAXN) X.gm[redo][lane] = X.W.t[lane];
                __syncwarp();
                if (SEL && B.sel && lane < n && count < B.sel_cap)
                    B.sel[((size_t)p * B.sel_cap + count) * MAXN + P.greedy.vert[lane]] = X.W.t[lane];
                use_maps(A.used + (size_t)s * B.G.words, A.dirty + (size_t)s * DIRTY_CAP, lane == redo, X.gm[lane], n, nd);
                count++;
                over = count >= cap;
            }
            todo &= ~(1u << redo);
        }
    }
    while (!over && !stopped) {
        if (m == 0) {
            // the finished groups from g on that fit a warp: m of them
            const int kg = lane / GS;
            const bool fin = lane > 0 && lane < 32 / GS && g + lane < ngroups &&
                             (cg(status + ((g + lane) & RM)) & G_DONE);
            m = __ffs(~(__ballot_sync(FULLMASK, fin) | 1u)) - 1;
            const size_t gi = (size_t)s * A.RG + ((g + kg) & RM);
            const bool mapped = kg < m && (cg(A.mask + gi) >> (lane % GS) & 1u);
            ep_fresh += __reduce_add_sync(FULLMASK, kg < m && lane % GS == 0 ? cg(A.status + gi) >> G_STEPS : 0u);
            if (mapped) {
                const int4 *src = reinterpret_cast<const int4 *>(A.maps + (gi * GS + lane % GS) * MAXN);
                int4 *dst = reinterpret_cast<int4 *>(X.gm[lane]);
                dst[0] = cg(src);
                dst[1] = cg(src + 1);
            }
            have = __ballot_sync(FULLMASK, mapped);
            todo = have;
            // (their searches were long ones)
            whole = __ballot_sync(FULLMASK, mapped && (cg(A.mask2 + gi) >> (lane % GS) & 1u));
            __syncwarp();
        }
        if (todo) {
            // maps in order up to the first stale one: stale when a vertex has been used, by an
            // earlier group or by an earlier map of this one
            bool bad = (todo >> lane & 1u) && !(have >> lane & 1u);
            const bool mapped = (todo & have) >> lane & 1u;
            int32_t mv[MAXN];  // this lane's map (entries past n equal no vertex)
#pragma unroll
            for (int l = 0; l < MAXN; l++) {
                mv[l] = mapped && l < n ? X.gm[lane][l] : -1;
                if (mapped && l < n) bad |= used_bit(used, mv[l]);
            }
            uint32_t take = 0, rem = todo;
            int redo = -1;
            while (rem) {
                const int i = __ffs(rem) - 1;
                rem &= rem - 1;
                if (__shfl_sync(FULLMASK, (int)bad, i)) {
                    redo = i;
                    break;
                }
                take |= 1u << i;
                if (count + __popc(take) >= cap) break;
                if (rem >> lane & 1u)
                    for (int l = 0; l < n; l++) {
                        const int32_t v = X.gm[i][l];
#pragma unroll
                        for (int k = 0; k < MAXN; k++) bad |= mv[k] == v;
                    }
            }
            if (take) {
                const bool mine = take >> lane & 1u;
                if (SEL && B.sel && mine) {
                    const int64_t at = count + __popc(take & ((1u << lane) - 1u));
                    if (at < B.sel_cap)
                        for (int l = 0; l < n; l++)
                            B.sel[((size_t)p * B.sel_cap + at) * MAXN + P.greedy.vert[l]] = X.gm[lane][l];
                }
                use_maps(A.used + (size_t)s * B.G.words, A.dirty + (size_t)s * DIRTY_CAP, mine, X.gm[lane], n, nd);
                count += __popc(take);
                todo &= ~take;
                over = count >= cap;
            }
            if (over || redo < 0) continue;
            if (!(whole >> redo & 1u)) {
                const uint32_t again = __ballot_sync(FULLMASK, bad) & todo & ~whole;
                if (lane == 0) {
                    RetireState &R = X.R;
                    R.count = count;
                    R.g = g; R.m = m; R.again = again;
                    R.lim = lim; R.window = window; R.ep_left = ep_left; R.nd = nd;
                    R.have = have; R.todo = todo; R.whole = whole; R.ep_fresh = ep_fresh; R.ep_again = ep_again;
                }
                __syncwarp();
                return RT_LANES;
            }
            // the root again, past its stale map (nothing before it can have become a map)
            root = __ldg(G.lab_vtx + rb + g * GS + redo);
            from = 0;
            bool go = !warp_used(used, root);
            if (go && (have >> redo & 1u)) {
                const bool u = lane < n && used_bit(used, X.gm[redo][lane]);
                if (lane < MAXN) X.W.t[lane] = X.gm[redo][lane];
                from = __ffs(__ballot_sync(FULLMASK, u)) - 1;
                if (from < 1) from = 1;
                __syncwarp();
            } else if (go) {
                go = level_fits(G, root, X.W.C[0]);
            }
            if (!go) {
                todo &= ~(1u << redo);
                continue;
            }
            if (lane == 0) {
                RetireState &R = X.R;
                R.count = count;
                R.g = g; R.m = m; R.redo = redo;
                R.lim = lim; R.window = window; R.ep_left = ep_left; R.nd = nd;
                R.have = have; R.todo = todo; R.whole = whole; R.ep_fresh = ep_fresh; R.ep_again = ep_again;
            }
            __syncwarp();
            return RT_SEARCH;
        }
        // the batch is retired
        const int head = g + m;
        // every selection to come needs a root of its own: below c the pattern is infrequent,
        // which is all mining asks
        const int64_t left = (int64_t)(re - rb) - (int64_t)head * GS;
        if (head >= ngroups || (P.decide_only && count + left < cap)) {
            over = true;
            break;
        }
        // the window, and the claim limit: at most the groups that the maps still wanted should
        // take at the rate seen so far, and a quarter more
        ep_left -= m;
        if (ep_left <= 0) {
            const uint32_t one = ep_fresh / (uint32_t)window + STREAM_REDO_STEPS;
            if (ep_again <= one) window = min(2 * window, A.RG);
            else if (ep_again > 4 * one) window = max(window / 2, 2);
            ep_left = window;
            ep_fresh = ep_again = 0;
        }
        int64_t want = window;
        if (cap != CAP_INF) {
            const float per = (float)head / (float)(count + 1);
            want = min(want, (int64_t)(1.25f * (float)(cap - count) * per) + 1);
        }
        const int32_t target = (int32_t)min((int64_t)ngroups, (int64_t)head + max(want, (int64_t)1));
        const int32_t delta = max(target - lim, 0);
        lim += delta;
        if (lane < m) atomicExch(status + ((g + lane) & RM), 0u);
        if (lane == 0) {
            T->count = count;
            T->head = head;
            T->lim = lim;
            T->window = window;
            T->ep_left = ep_left;
            T->ep_fresh = ep_fresh;
            T->ep_again = ep_again;
            T->ndirty = nd;
        }
        __threadfence();
        __syncwarp();
        uint32_t old = 0;
        if (lane == 0) {
            if (delta > 0) atomicAdd(A.words + s, (unsigned long long)delta);
            old = atomicOr(status + (head & RM), G_HEAD);
        }
        old = __shfl_sync(FULLMASK, old, 0);
        if (!(old & G_DONE)) return RT_DONE;  // its warp will find the HEAD bit
        g = head;
        m = 0;
    }
    if (lane == 0) {
        T->count = count;
        T->head = g;
        T->ndirty = nd;
    }
    if (over) mark_done(A, s);
    __syncwarp();
    return RT_DONE;
}

// M_TASK: a part of a shared search; M_ROOT: one root of a shared group.
enum : int { M_CLAIM, M_GROUP, M_RETIRE, M_TASK, M_ROOT };

// Share the roots `todo` of group g, left open by the lanes: a task each.  The warp that finishes the last
// one publishes the group.  False (nothing changed) when there is no room.
__device__ __noinline__ bool share_roots(const Batch &B, const StreamArgs &A, int s, int p, int g, uint32_t todo,
                                         uint32_t found, uint32_t gsteps) {
    const int lane = threadIdx.x & 31;
    const int n = __popc(todo), n0 = min(n, TASK_CUT), n1 = n - n0;
    int b0 = -1, b1 = -1, tm = -1;
    if (lane == 0) {
        b0 = take_index(&B.ctl->blocks_free, A.block_next, &B.ctl->blocks_bump, STREAM_TASKS / TASK_CUT);
        if (b0 >= 0 && n1) b1 = take_index(&B.ctl->blocks_free, A.block_next, &B.ctl->blocks_bump, STREAM_TASKS / TASK_CUT);
        if (b0 >= 0 && (b1 >= 0 || !n1)) tm = take_index(&B.ctl->teams_free, A.team_next, &B.ctl->teams_bump, STREAM_TEAMS);
        if (tm < 0) {
            if (b0 >= 0) stack_push(&B.ctl->blocks_free, A.block_next, b0);
            if (b1 >= 0) stack_push(&B.ctl->blocks_free, A.block_next, b1);
        } else {
            StreamTeam *T = team_of(A, tm);
            T->open = n;
            T->s = s; T->p = p; T->g = g;
            T->found = found; T->found2 = 0; T->gsteps = gsteps;
            A.block_open[b0] = n0;
            if (n1) A.block_open[b1] = n1;
        }
    }
    tm = __shfl_sync(FULLMASK, tm, 0);
    b0 = __shfl_sync(FULLMASK, b0, 0);
    b1 = __shfl_sync(FULLMASK, b1, 0);
    if (tm < 0) return false;
    if (lane < n) {
        const int t = lane < n0 ? b0 * TASK_CUT + lane : b1 * TASK_CUT + lane - n0;
        uint32_t *dst = A.tasks + (size_t)t * STREAM_TASK_WORDS;
        dst[TASK_TEAM] = (uint32_t)tm;
        dst[TASK_KEY] = __fns(todo, 0, lane + 1);
        dst[TASK_KEY + 1] = 0u;
        dst[TASK_SHIFT] = SHIFT_ROOT;
    }
    if (n1) ready_put(B, A, b1 * TASK_CUT, n1);
    ready_put(B, A, b0 * TASK_CUT, n0);
    return true;
}

// Cut the suspended search in X.W: its tasks go to the ready stack.  `team` < 0: a new team, to go on
// with (mode, s, p, g, i, todo, found, found2, gsteps) and X.R, X.gm when the search is decided; otherwise the
// search is a task of that team with this key.  False (nothing changed) when it cannot be cut: no
// open level, keys or room.
__device__ __noinline__ bool cut_search(const Batch &B, const StreamArgs &A, StreamWarp &X, int team,
                                        unsigned long long key, int shift, int mode, int s, int p, int g, int i,
                                        uint32_t todo, uint32_t found, uint32_t found2, uint32_t gsteps) {
    const int lane = threadIdx.x & 31;
    WarpState &W = X.W;
    const int lvl0 = W.level, floor0 = W.floor;
    int m = -1;
    for (int l = floor0; l <= lvl0; l++)
        if (W.pos[l] < W.hi[l]) {
            m = l;
            break;
        }
    if (m < 0 || shift < KEY_CUT) return false;
    const uint32_t a = W.pos[m], b = W.hi[m], len = b - a, mask_m = W.mask[m], conf_m = W.conf[m];
    const int pieces = (int)min(len, (uint32_t)(TASK_CUT - 2)), nt = pieces + 2;
    int blk = -1, tm = team;
    if (lane == 0) {
        blk = take_index(&B.ctl->blocks_free, A.block_next, &B.ctl->blocks_bump, STREAM_TASKS / TASK_CUT);
        if (blk >= 0 && team < 0) {
            tm = take_index(&B.ctl->teams_free, A.team_next, &B.ctl->teams_bump, STREAM_TEAMS);
            if (tm < 0) {
                stack_push(&B.ctl->blocks_free, A.block_next, blk);
                blk = -1;
            }
        }
    }
    blk = __shfl_sync(FULLMASK, blk, 0);
    tm = __shfl_sync(FULLMASK, tm, 0);
    if (blk < 0) return false;
    StreamTeam *T = team_of(A, tm);
    if (lane == 0) A.block_open[blk] = nt;
    if (team < 0) {
        if (lane == 0) {
            T->best = ~0ull;
            T->open = nt;
            T->s = s; T->p = p; T->g = g; T->mode = mode; T->i = i;
            T->todo = todo; T->found = found; T->found2 = found2; T->gsteps = gsteps;
        }
        const uint32_t *src = reinterpret_cast<const uint32_t *>(&X.R);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&T->R);
        for (int k = lane; k < (int)(sizeof(RetireState) / 4); k += 32) dst[k] = src[k];
        for (int l = 0; l < MAXN; l++) T->gm[lane][l] = X.gm[lane][l];
    } else if (lane == 0) {
        atomicAdd(&T->open, nt - 1);
    }
    const int t0 = blk * TASK_CUT;
    const int sub = shift - KEY_CUT;
    for (int j = 0; j < nt; j++) {
        __syncwarp();
        if (lane == 0) {
            if (j == 0) {  // what the search has begun of level m, nothing more
                W.level = lvl0;
                W.floor = m;
                W.pos[m] = a;
                W.hi[m] = a;
                W.mask[m] = mask_m;
                W.conf[m] = conf_m;
            } else if (j <= pieces) {  // candidates [a + len (j-1) / pieces, a + len j / pieces) of level m
                W.level = m;
                W.mask[m] = 0;
                W.floor = m;
                W.pos[m] = a + (uint32_t)((uint64_t)len * (j - 1) / pieces);
                W.hi[m] = a + (uint32_t)((uint64_t)len * j / pieces);
                W.conf[m] = 0;
            } else {  // the rest: level m exhausted, plain backtracking below it
                W.level = m;
                W.mask[m] = 0;
                W.floor = floor0;
                W.pos[m] = b;
                W.hi[m] = b;
                W.conf[m] = (1u << m) - 1u;
            }
        }
        __syncwarp();
        uint32_t *dst = A.tasks + (size_t)(t0 + j) * STREAM_TASK_WORDS;
        for (int w = lane; w < DFS_SAVE_WORDS; w += 32) dst[w] = reinterpret_cast<const uint32_t *>(&W)[w];
        if (lane == 0) {
            const unsigned long long k = key + ((unsigned long long)j << sub);
            dst[TASK_TEAM] = (uint32_t)tm;
            dst[TASK_KEY] = (uint32_t)k;
            dst[TASK_KEY + 1] = (uint32_t)(k >> 32);
            dst[TASK_SHIFT] = (uint32_t)sub;
        }
    }
    ready_put(B, A, t0, nt);
    return true;
}

// Two resident blocks take an SM's registers, and the launch lasts as long as its heaviest pattern: on all SMs it
// would hold up every other stream of the process, servers among them, for hundreds of milliseconds.  So
// one SM in 76 is left alone, one in 8 while the graph has a server: a block that finds itself on one of the
// last SMs leaves as soon as all but A.spare of the blocks run elsewhere.  (It does not leave at once: while another kernel holds the
// other SMs, the free places would be these, and every block would pass through them.  When that kernel
// goes on for SPARE_WAIT, it stays.)  Whole SMs, because a kernel that needs more shared memory than this one
// left it cannot start on a shared SM.  And a block whose warps have all been idle for about a millisecond leaves, but for a quarter of the grid: what
// becomes ready later is found by the warp that made it ready, if by no other.
//
// Requests of a server on another graph beside a batch of 4,000 on 100k vertices: p50 88 ms and p99 270 when
// all SMs were held, 0.8 and 2.8 with 2 of 152 SMs free (0.7 and 4.3 beside windowed rounds).  Blocks that
// leave cost nothing; deep mining, which fills the chip, takes 0.7 % longer with 2 SMs free, 1.8 % with 4
// and 2.7 % with 8.  A stream of heavy requests, though, ends at 71 ms with 8 SMs, 83 with 4 and 90
// with 2 (77 beside windowed rounds), hence the more SMs for a graph that is being served.
//
// (128 registers a thread: with 64 and twice the warps the same work took up to half as long again, the
// kernel's spills and its misses of the instruction cache -- a third of the warps' time then -- grew.)
template <class View>
__global__ void __launch_bounds__(SEARCH_THREADS, STREAM_BLOCKS) k_stream(const __grid_constant__ Batch B,
                                                                         const __grid_constant__ StreamArgs A) {
    const View &G = static_cast<const View &>(B.G);
    __shared__ StreamWarp ws[STREAM_WARPS];
    __shared__ int s_block, s_idle;  // number among the blocks that stay; warps idle for long
    if (threadIdx.x == 0) {
        int b = (int)blockIdx.x;
        if (A.spare) {
            uint32_t sm;
            asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
            bool leave = false;
            if ((int)sm >= A.spare_sm) {
                const unsigned long long t0 = global_ns();
                for (;;) {
                    leave = *reinterpret_cast<volatile int32_t *>(&B.ctl->arrived) >= (int)gridDim.x - A.spare;
                    if (leave || global_ns() - t0 > SPARE_WAIT) break;
                    __nanosleep(STREAM_NAP);
                }
            }
            b = leave ? -1 : atomicAdd(&B.ctl->arrived, 1);
        }
        s_block = b;
        s_idle = 0;
    }
    __syncthreads();
    const int block = s_block;
    if (block < 0) return;
    const int lane = threadIdx.x & 31;
    StreamWarp &X = ws[threadIdx.x >> 5];
    const int gw = (int)((block * blockDim.x + threadIdx.x) >> 5);
    const int nw = (int)(((gridDim.x - A.spare) * blockDim.x) >> 5);
    if (lane == 0) X.W.acc_scanned = X.W.acc_bound = X.W.acc_maps = X.W.acc_items = 0;
    __syncwarp();
    for (int s = gw; s < A.S; s += nw) start_slot(B, A, s);
    // The first STREAM_HOME warps of a slot stay with it while it has work and look at its claim
    // word often; all others roam: they look over the slots at growing intervals.  (Thousands of
    // warps polling at full speed slowed every load of the searching ones several times over.)
    const int home = gw / A.S < STREAM_HOME ? gw % A.S : -1;
    const int leave_polls = home >= 0 ? LEAVE_POLLS_HOME : LEAVE_POLLS;
    int s = gw % A.S, idle = 0, cur_p = -1;
    uint32_t nap = STREAM_NAP;
    int mode = M_CLAIM;
    // the group being searched
    int g = 0, p = 0, i = 0;
    uint32_t todo = 0, found = 0, found2 = 0, gsteps = 0;  // found2: by the whole warp
    int res = -1, why = STOP_NO;
    // the task being searched
    int task = -1, team = -1, gteam = -1, shift = KEY_BITS;  // gteam: the team of a shared group
    unsigned long long key = 0;
    for (;;) {
        if (mode == M_CLAIM) {
            if (late(B)) break;
            int nr = 0;
            if (lane == 0) nr = *reinterpret_cast<volatile int32_t *>(&B.ctl->n_ready);
            const int tk = __shfl_sync(FULLMASK, nr, 0) > 0 ? ready_take(B, A, gw) : -1;
            g = tk >= 0 ? 0 : claim(A, s);
            if (g < 0) {
                // (the batch's state is one line that every warp looks at: as seldom as possible)
                // (a home warp whose slot has no more patterns looks each time)
                bool look = home < 0 || (idle & 7) == 7;
                if (!look) {
                    if (lane == 0) look = word_of(A.words + s) == 0ull;
                    look = __any_sync(FULLMASK, look);
                }
                if (look) {
                    const int t = find_slot(A, s);
                    if (t >= 0) {
                        s = t;
                        g = claim(A, s);
                    } else {
                        bool end = false;
                        if (lane == 0)
                            end = *reinterpret_cast<volatile int32_t *>(&B.ctl->done_count) >= B.P ||
                                  *reinterpret_cast<volatile int32_t *>(&B.ctl->expired);
                        if (__any_sync(FULLMASK, end)) break;
                    }
                }
                if (g < 0) {
                    if (idle == 0 && lane == 0) atomicAdd(&B.ctl->idlers, 1);
                    if (++idle > IDLE_POLLS) break;
                    if (block >= A.keep && idle >= leave_polls) {
                        bool all = false;
                        if (lane == 0) {
                            if (idle == leave_polls) atomicAdd(&s_idle, 1);
                            all = *reinterpret_cast<volatile int *>(&s_idle) >= STREAM_WARPS;
                        }
                        if (__any_sync(FULLMASK, all)) break;
                    }
                    if (home >= 0) s = home;
                    __nanosleep(nap);
                    nap = min(nap + nap / 2, home >= 0 ? STREAM_NAP_HOME : STREAM_NAP_MAX);
                    continue;
                }
            }
            if (idle > 0 && lane == 0) {
                atomicSub(&B.ctl->idlers, 1);
                if (block >= A.keep && idle >= leave_polls) atomicSub(&s_idle, 1);
            }
            nap = STREAM_NAP;
            idle = 0;
            if (tk >= 0) {
                task = tk;
                const uint32_t *src = A.tasks + (size_t)tk * STREAM_TASK_WORDS;
                team = (int)cg(src + TASK_TEAM);
                key = (unsigned long long)cg(src + TASK_KEY + 1) << 32 | cg(src + TASK_KEY);
                shift = (int)cg(src + TASK_SHIFT);
                const StreamTeam *T = team_of(A, team);
                s = cg(&T->s);
                p = cg(&T->p);
                if (p != cur_p) {
                    const Plan &P = B.plans[p];
                    load_level_plan(X.W, P.greedy, P);
                    cur_p = p;
                }
                if (shift == SHIFT_ROOT) {
                    gteam = team;
                    g = cg(&T->g);
                    i = (int)key;
                    mode = M_ROOT;
                } else {
                    __syncwarp();
                    for (int w = lane; w < DFS_SAVE_WORDS; w += 32) reinterpret_cast<uint32_t *>(&X.W)[w] = cg(src + w);
                    __syncwarp();
                    mode = M_TASK;
                }
            }
        }
        uint32_t lmask = 0;  // roots (counted from lbase) that the lanes search now
        int lbase = 0;
        if (mode == M_CLAIM) {
            const StreamSlot *T = A.slots + s;
            const int re = cg(&T->root_end);
            lbase = cg(&T->root_begin) + g * A.GS;
            p = cg(&T->p);
            if (p != cur_p) {
                const Plan &P = B.plans[p];
                load_level_plan(X.W, P.greedy, P);
                cur_p = p;
            }
            lmask = __ballot_sync(FULLMASK, lane < A.GS && lbase + lane < re);
        }
        int32_t root = 0;
        uint2 fs = make_uint2(0u, 0u);
        int from = 0;
        const int ring = g & (A.RG - 1);
        bool release = false;
        if (mode == M_GROUP || mode == M_ROOT) {
            if (todo || mode == M_ROOT) {
                if (mode == M_GROUP) {
                    i = __ffs(todo) - 1;
                    todo &= todo - 1;
                }
                root = __ldg(G.lab_vtx + cg(&A.slots[s].root_begin) + g * A.GS + i);
                fs = lane_slice(G, root, X.W.L.lab[1], X.W.L.bdir[1] & 3u);
            } else {
                // publish the group; retire if it is the head.  An aborted search means that the
                // pattern is finished or the deadline has passed: nothing to publish.
                release = true;
                if (why != STOP_ABORT) {
                    const size_t gi = (size_t)s * A.RG + ring;
                    if (lane == 0) {
                        A.mask[gi] = found;
                        A.mask2[gi] = found2;
                    }
                    __threadfence();
                    __syncwarp();
                    uint32_t old = 0;
                    if (lane == 0) old = atomicOr(A.status + gi, G_DONE | min(gsteps, G_STEPS_MAX) << G_STEPS);
                    if (__shfl_sync(FULLMASK, old, 0) & G_HEAD) {
                        retire_begin(A, X, s, g);
                        res = -1;
                        mode = M_RETIRE;
                        release = false;
                    }
                }
            }
        }
        if (mode == M_RETIRE) {
            // (a retiring warp may go on for many batches of roots that lanes search again)
            if (res == RES_LANES && late(B)) break;
            const int rt = retire_step(G, B, A, X, s, res, root, from);
            if (rt == RT_DONE) {
                release = true;
            } else if (rt == RT_LANES) {
                lbase = X.R.rb + X.R.g * A.GS;
                lmask = X.R.again;
            } else if (from == 0) {
                fs = lane_slice(G, root, X.W.L.lab[1], X.W.L.bdir[1] & 3u);
            }
        }
        if (mode == M_CLAIM || lmask) {
            int32_t r = -1;
            uint2 first = make_uint2(0u, 0u);
            bool ok = false;
            if (lmask >> lane & 1u) {
                r = __ldg(G.lab_vtx + lbase + lane);
                first = lane_slice(G, r, X.W.L.lab[1], X.W.L.bdir[1] & 3u);
                const bool fits = level_fits(G, r, X.W.C[0]);
                ok = !used_bit(A.used + (size_t)s * G.words, r) && fits && first.x != first.y;
            }
            const int nsearch = __popc(__ballot_sync(FULLMASK, ok));
            SearchWork work;
            uint32_t open = 0, its = 0;
            const uint32_t got = lane_searches(G, X, A.used + (size_t)s * G.words, A.dead + ((size_t)s << DEAD_LOG), ok,
                                               r, first, open, its, work);
            if (lane == 0) {
                X.W.acc_scanned += work.scanned;
                X.W.acc_bound += work.bound;
                X.W.acc_maps += (unsigned)(__popc(got) * X.W.n);
                X.W.acc_items += (unsigned)(nsearch - __popc(open));
                atomicAdd(&B.st[p].steps, (unsigned long long)its);
                if (mode == M_CLAIM && nsearch)
                    atomicAdd((unsigned long long *)&B.st[p].searched, (unsigned long long)nsearch);
            }
            if (mode == M_RETIRE) {
                if (lane == 0) {
                    X.R.got = got;
                    X.R.left = open;
                    X.W.last_steps = its;
                }
                __syncwarp();
                res = RES_LANES;
                continue;
            }
            why = STOP_NO;
            found = got;
            found2 = 0;
            todo = open;
            gsteps = its;
            // (one lane looks: the bit may be set meanwhile, and the warp has to agree)
            uint32_t hd = 0;
            if (lane == 0) hd = cg(A.status + (size_t)s * A.RG + (g & (A.RG - 1))) & G_HEAD;
            // several open roots and warps without work: the roots are shared, at the head too (one after
            // another there they held up everything behind them)
            int il = 0;
            if (lane == 0 && __popc(todo) > 1 &&
                __popc(todo) * *reinterpret_cast<volatile uint32_t *>(&A.slots[s].last_steps) >= SHARE_STEPS)
                il = *reinterpret_cast<volatile int32_t *>(&B.ctl->idlers);
            const bool share = __shfl_sync(FULLMASK, il, 0) >= SPLIT_IDLE;
            if (__shfl_sync(FULLMASK, hd, 0) && !share) {
                // the head: what the lanes found is retired at once, the open roots in their turn
                retire_begin(A, X, s, g);
                if (lane == 0) {
                    X.R.m = 1;
                    X.R.have = found;
                    X.R.todo = found | todo;
                    X.R.whole = todo;
                    X.R.ep_fresh += gsteps;
                }
                __syncwarp();
                res = -1;
                mode = M_RETIRE;
            } else {
                const size_t gi = (size_t)s * A.RG + (g & (A.RG - 1));
                if (found >> lane & 1u) {
                    const int4 *src = reinterpret_cast<const int4 *>(X.gm[lane]);
                    int4 *dst = reinterpret_cast<int4 *>(A.maps + (gi * A.GS + lane) * MAXN);
                    dst[0] = src[0];
                    dst[1] = src[1];
                }
                __threadfence();
                __syncwarp();
                mode = share && share_roots(B, A, s, p, g, todo, found, gsteps) ? M_CLAIM : M_GROUP;
            }
            continue;
        }
        if (release) {
            // Whoever ends the pattern clears what this warp wrote for it (dead candidates, maps): every lane's
            // stores come before the reference falls.  An aborted search gets here with no fence of its own.
            __threadfence();
            __syncwarp();
            unsigned long long w = 0;
            if (lane == 0) w = atomicAdd(A.words + s, 0ull - W_REF1);
            w = __shfl_sync(FULLMASK, w, 0);
            if ((w & W_DONE) && ((w >> W_REFS) & W_REFMASK) == 1ull) end_slot(B, A, s, (int)((w >> W_NEXT) & W_FIELD));
            mode = M_CLAIM;
            continue;
        }
        // one root search: from the start, past the stale map in W.t whose first used vertex is at level
        // `from`, or a task of a shared one
        SearchWork work;
        unsigned long long bytes = 0;  // touched-bytes counts are not kept here
        uint32_t probes = 0, steps = 0, split_at = SPLIT_STEPS;
        if (mode != M_TASK) {
            key = 0;
            shift = KEY_BITS;
        }
        if (from > 0) state_of_map(G, X.W, from, bytes, probes);
        bool shared = false, nested = false;  // cut; into a team below this task
        for (bool again = from > 0 || mode == M_TASK;; again = true) {
            why = STOP_NO;
            res = dfs_run<StreamStop, true>(G, X.W, A.used + (size_t)s * G.words, root, bytes, probes, steps, again,
                                            work, StreamStop{A.words + s, mode == M_TASK ? &team_of(A, team)->best : nullptr,
                                                             key, B.ctl, B.deadline_ns, steps + STOP_EVERY, split_at, &why},
                                            fs, A.dead + ((size_t)s << DEAD_LOG));
            if (res != DFS_SUSPENDED || why != STOP_SPLIT) break;
            // what to go on with when a new team has decided it; a task whose key cannot be divided any more
            // gets a team of its own
            int tm = -1, back_i = i;
            uint32_t back[4] = {todo, found, found2, gsteps};
            if (mode == M_ROOT) {
                back[1] = (uint32_t)gteam;
                back[2] = (uint32_t)task;
            } else if (mode == M_TASK && shift >= KEY_CUT) {
                tm = team;
            } else if (mode == M_TASK) {
                nested = true;
                back_i = shift;
                back[0] = (uint32_t)key;
                back[1] = (uint32_t)team;
                back[2] = (uint32_t)task;
                back[3] = (uint32_t)(key >> 32);
            }
            shared = cut_search(B, A, X, tm, nested ? 0ull : key, nested ? KEY_BITS : shift, mode, s, p, g, back_i, back[0],
                                back[1], back[2], back[3]);
            if (shared) break;
            nested = false;
            split_at = steps + SPLIT_AGAIN;
        }
        if (lane == 0) {
            X.W.acc_scanned += work.scanned;
            X.W.acc_bound += work.bound;
            if (res == DFS_FOUND) X.W.acc_maps += (unsigned)X.W.n;
            X.W.acc_items++;
            X.W.last_steps = steps;
            atomicAdd(&B.st[p].steps, (unsigned long long)steps);
            atomicMax(&B.st[p].max_steps, steps);
            if (mode != M_TASK) *reinterpret_cast<volatile uint32_t *>(&A.slots[s].last_steps) = steps;
        }
        __syncwarp();
        bool parked = false;  // the search goes on elsewhere
        while (shared || mode == M_TASK) {
            bool last = false;
            if (mode == M_TASK && !nested) {
                // the task is finished, or has been replaced by its own tasks
                StreamTeam *T = team_of(A, team);
                if (!shared && res == DFS_FOUND && lane < MAXN)
                    A.tasks[(size_t)task * STREAM_TASK_WORDS + lane] = (uint32_t)X.W.t[lane];
                __threadfence();
                __syncwarp();
                if (lane == 0) {
                    int drop = task;
                    if (!shared && res == DFS_FOUND) {
                        const unsigned long long mine = key << 16 | (unsigned)task;
                        const unsigned long long old = atomicMin(&T->best, mine);
                        if (old > mine) drop = old == ~0ull ? -1 : (int)(old & 0xFFFFu);
                    }
                    if (drop >= 0) drop_task(B, A, drop);
                    if (!shared) {
                        __threadfence();
                        last = atomicSub(&T->open, 1) == 1;
                    }
                }
                last = __any_sync(FULLMASK, last);
            }
            if (!last) {
                parked = true;
                break;
            }
            // the shared search is decided: go on with what it belongs to
            __threadfence();
            StreamTeam *T = team_of(A, team);
            mode = cg(&T->mode);
            g = cg(&T->g);
            i = cg(&T->i);
            todo = cg(&T->todo);
            found = cg(&T->found);
            found2 = cg(&T->found2);
            if (mode == M_ROOT) {
                gteam = (int)found;
                task = (int)found2;
            }
            gsteps = cg(&T->gsteps);
            const uint32_t *src = reinterpret_cast<const uint32_t *>(&T->R);
            for (int k = lane; k < (int)(sizeof(RetireState) / 4); k += 32) reinterpret_cast<uint32_t *>(&X.R)[k] = cg(src + k);
            for (int l = 0; l < MAXN; l++) X.gm[lane][l] = cg(&T->gm[lane][l]);
            const unsigned long long best = cg(&T->best);
            why = STOP_NO;
            res = DFS_NONE;
            if (best != ~0ull) {
                const int tk = (int)(best & 0xFFFFu);
                if (lane < MAXN) X.W.t[lane] = (int32_t)cg(A.tasks + (size_t)tk * STREAM_TASK_WORDS + lane);
                res = DFS_FOUND;
                __syncwarp();
                if (lane == 0) drop_task(B, A, tk);
            } else {
                bool end = false;
                if (lane == 0)
                    end = (word_of(A.words + s) & W_DONE) || *reinterpret_cast<volatile int32_t *>(&B.ctl->expired);
                if (__any_sync(FULLMASK, end)) {
                    res = DFS_SUSPENDED;
                    why = STOP_ABORT;
                }
            }
            __syncwarp();
            if (lane == 0) stack_push(&B.ctl->teams_free, A.team_next, team);
            __syncwarp();
            shared = nested = false;
            if (mode == M_TASK) {
                team = (int)found;
                task = (int)found2;
                key = (unsigned long long)gsteps << 32 | todo;
                shift = i;
            }
        }
        if (parked) {
            mode = M_CLAIM;
            continue;
        }
        if (mode == M_RETIRE) continue;
        if (mode == M_ROOT) {
            // a root of a shared group: its map and bits; the last one publishes the group
            StreamTeam *T = team_of(A, gteam);
            if (res == DFS_FOUND && lane < MAXN)
                A.maps[(((size_t)s * A.RG + (g & (A.RG - 1))) * A.GS + i) * MAXN + lane] = X.W.t[lane];
            __threadfence();
            __syncwarp();
            bool last = false, end = false;
            if (lane == 0) {
                if (res == DFS_FOUND) {
                    atomicOr(&T->found, 1u << i);
                    atomicOr(&T->found2, 1u << i);
                }
                atomicAdd(&T->gsteps, steps);
                drop_task(B, A, task);
                __threadfence();
                last = atomicSub(&T->open, 1) == 1;
                end = (word_of(A.words + s) & W_DONE) || *reinterpret_cast<volatile int32_t *>(&B.ctl->expired);
            }
            if (!__any_sync(FULLMASK, last)) {
                mode = M_CLAIM;
                continue;
            }
            __threadfence();
            found = cg(&T->found);
            found2 = cg(&T->found2);
            gsteps = cg(&T->gsteps);
            todo = 0;
            why = __any_sync(FULLMASK, end) ? STOP_ABORT : STOP_NO;
            mode = M_GROUP;
            __syncwarp();
            if (lane == 0) stack_push(&B.ctl->teams_free, A.team_next, gteam);
            __syncwarp();
            continue;
        }
        gsteps += steps;
        if (res == DFS_FOUND) {
            const size_t gi = (size_t)s * A.RG + (g & (A.RG - 1));
            if (lane < MAXN) A.maps[(gi * A.GS + i) * MAXN + lane] = X.W.t[lane];
            found |= 1u << i;
            found2 |= 1u << i;
            __syncwarp();
        } else if (res == DFS_SUSPENDED) {
            todo = 0;
        }
    }
    if (idle > 0 && lane == 0) atomicSub(&B.ctl->idlers, 1);
    if (lane == 0 && X.W.acc_items) {
        atomicAdd(&B.ctl->bytes_greedy, 4ull * X.W.acc_scanned + 8ull * X.W.acc_bound + 4ull * X.W.acc_maps);
        atomicAdd(&B.ctl->alg_scanned, X.W.acc_scanned);
        atomicAdd(&B.ctl->alg_bound, X.W.acc_bound);
        atomicAdd(&B.ctl->alg_map_words, X.W.acc_maps);
        atomicAdd(&B.ctl->search_items, X.W.acc_items);
    }
}

// After a deadline: slots still active give their patterns the maps committed so far, and every
// pattern still in its greedy phase is stopped.
__global__ void k_stream_expire_slots(const __grid_constant__ Batch B, const __grid_constant__ StreamArgs A) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (!B.ctl->expired || s >= A.S || !(A.words[s] & W_ACTIVE)) return;
    const StreamSlot &T = A.slots[s];
    B.st[T.p].count = T.count;
}

__global__ void k_stream_expire(const __grid_constant__ Batch B) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (!B.ctl->expired || p >= B.P) return;
    PatState &S = B.st[p];
    if (S.phase != PH_GREEDY) return;
    if (B.sel) S.logged = (int32_t)min(min(S.count, B.plans[p].cap), (int64_t)B.sel_cap);
    S.cancelled = 1;
    S.done = 1;
    S.phase = PH_MNI;
}

}  // namespace

int stream_blocks_per_sm() {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_stream<DevGraphView>, SEARCH_THREADS, 0) != cudaSuccess) per_sm = 1;
    return per_sm < 1 ? 1 : per_sm;
}

void launch_stream(const Batch &B, const StreamArgs &A, bool fast, int blocks, cudaStream_t stream) {
    if (fast)
        k_stream<FastView><<<blocks, SEARCH_THREADS, 0, stream>>>(B, A);
    else
        k_stream<DevGraphView><<<blocks, SEARCH_THREADS, 0, stream>>>(B, A);
}

void launch_stream_expire(const Batch &B, const StreamArgs &A, cudaStream_t stream) {
    k_stream_expire_slots<<<(A.S + 255) / 256, 256, 0, stream>>>(B, A);
    k_stream_expire<<<(B.P + 255) / 256, 256, 0, stream>>>(B);
}

}  // namespace fx

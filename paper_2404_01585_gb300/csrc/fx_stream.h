// Streaming greedy (stream.cu): one launch that takes every pattern of a batch through its greedy
// phase.  Host-side interface used by the batch driver (kernels.cu).
#pragma once
#include "fx_batch.cuh"

namespace fx {

// One slot: the pattern it is working on.  Fields are read and written by the slot's retiring
// warp (one at a time; the role is handed on through the group status words) and by the warp that
// starts or ends the pattern, which is alone on the slot.
struct alignas(128) StreamSlot {
    int64_t count;        // maps selected
    int32_t p;            // pattern
    int32_t root_begin, root_end;
    int32_t ngroups;      // groups of GS consecutive roots
    int32_t head;         // first group not retired
    int32_t lim;          // groups below this one may be claimed
    int32_t window;       // groups past the head that may be in flight
    int32_t ep_left;      // the epoch that adapts the window: groups left,
    uint32_t ep_fresh, ep_again;  // chunks of first searches and of searches past a stale map
    int32_t ndirty;       // used-bitmap words made non-zero (listed up to DIRTY_CAP)
    uint32_t last_steps;  // chunks of the last search by a whole warp (any warp writes it; a hint)
};

struct StreamArgs {
    int32_t S;            // slots
    int32_t GS;           // roots per group (a power of two <= STREAM_GS_MAX)
    int32_t RG;           // ring length in groups (a power of two)
    int32_t window0;      // groups in flight at the start of a pattern
    unsigned long long *words;  // [S] claim words
    StreamSlot *slots;    // [S]
    uint32_t *status;     // [S][RG] group status bits, and the chunks scanned
    uint32_t *mask, *mask2;  // [S][RG] roots of the group with a map; those found by long searches
    int32_t *maps;        // [S][RG][GS][MAXN] their maps, by level
    uint32_t *used;       // [S][words] used bitmaps, all zero between launches
    int32_t *dirty;       // [S][DIRTY_CAP]
    uint32_t *dead;       // [S][1 << DEAD_LOG] dead candidates, all zero between launches
    uint32_t *tasks;      // [STREAM_TASKS][STREAM_TASK_WORDS] saved sub-searches of shared searches
    int32_t *task_next, *block_next, *block_open;  // their links; of their blocks: links, tasks open
    unsigned char *teams; // [STREAM_TEAMS][STREAM_TEAM_BYTES] shared searches
    int32_t *team_next;
    // SMs left to other work (see k_stream): SMs from spare_sm on, the blocks that fit on them
    int32_t spare, spare_sm;
    int32_t keep;         // blocks below it stay to the end of the batch
};

constexpr int STREAM_GS_MIN = 4, STREAM_GS_MAX = 32;
constexpr int64_t STREAM_BITMAP_BYTES = 2ll << 30;  // used bitmaps of all slots, at most
constexpr int64_t STREAM_RING_ROOTS = 1 << 20;      // roots in flight over all slots, at most
constexpr int64_t STREAM_RING_SLOT_MIN = 128, STREAM_RING_SLOT_MAX = 16384;  // ... of one slot
constexpr int STREAM_SLOT_WARPS = 512;
constexpr int STREAM_SPARE_DIV = 76, STREAM_SPARE_DIV_SERVED = 8;  // one in so many SMs is left to other work
constexpr int STREAM_KEEP_DIV = 4;    // a quarter of a full grid stays to the end
constexpr int STREAM_TASKS = 8192, STREAM_TASK_WORDS = 192, STREAM_TEAMS = 1024, STREAM_TEAM_BYTES = 1280;

int stream_blocks_per_sm();
// Whether the kernel for graphs with all their tables runs; `cyclic`: some pattern has a cycle.
inline bool stream_fast(const Batch &B, bool cyclic) { return B.G.off && (B.G.edges || !cyclic) && !B.sel; }
void launch_stream(const Batch &B, const StreamArgs &A, bool fast, int blocks, cudaStream_t stream);
// After the stream kernel: when the deadline passed, the patterns it left undecided.
void launch_stream_expire(const Batch &B, const StreamArgs &A, cudaStream_t stream);

}  // namespace fx

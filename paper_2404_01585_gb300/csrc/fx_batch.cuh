// Device state of a batch evaluation, shared by the windowed rounds (kernels.cu) and the streaming
// greedy (stream.cu): per-pattern state, control words, the batch view, saved-search layout.
#pragma once
#include "fx_kern.cuh"

namespace fx {

// window slot states.  A SEQ slot's root search ran out of its per-round budget: its remaining
// search space is an ordered list of saved sub-searches (the first one's index in the slot's
// map entry 0, each saved state holding the index of the next); the slot's map is the map of
// the first sub-search in that order that finds one, once every earlier one has found none.
enum : int32_t { SLOT_NEEDS = 0, SLOT_MAP = 1, SLOT_NONE = 2, SLOT_SEQ = 3 };
// saved sub-search status (word SUSP_STATUS of its saved state); its map in SUSP_MAP..+7
enum : int32_t { SS_PENDING = 0, SS_NONE = 1, SS_FOUND = 2 };
constexpr int SPLIT_MAX = 15;  // pieces one split may create


// slot phases: free, greedy rounds, MNI pending, result ready
enum : int32_t { PH_FREE = 0, PH_GREEDY = 1, PH_MNI = 2, PH_READY = 3 };

struct PatState {
    int64_t count;     // maps selected so far
    int64_t searched;  // root searches run
    int32_t cursor;    // next root (index into lab_vtx)
    int32_t nwin;      // slots in the window
    int32_t W;         // target window size
    int32_t done;
    int32_t exhausted; // every root processed
    int32_t rounds;
    int32_t phase;
    int32_t logged;    // selected maps written to the selection log
    unsigned long long mni_cnt[MAXN];
    unsigned long long steps;  // candidate chunks scanned by the greedy searches
    uint32_t max_steps;        // largest chunk count of one greedy search
    int32_t buf;               // current window buffer (0 or 1)
    uint32_t susp_mask;        // saved-search slots in use (KSUSP bits)
    uint32_t cancelled;        // stopped at a deadline before its decision
    uint32_t mni_cut;          // the MNI pass passed the deadline before this pattern's count
    int32_t ndirty;            // used-bitmap words this pattern made non-zero (listed up to DIRTY_CAP)
};

constexpr int READY_STACKS = 64;  // streaming greedy: stacks of tasks ready to run

struct Ctl {
    int32_t n_items[2];
    int32_t next_item[2];
    int32_t active[2];
    int32_t acount[2];    // lengths of the two active-pattern lists
    int32_t idle[2];      // warps of the search launch that found no work item left
    int32_t drain[2];     // set once idle reaches the launch's drain threshold
    int32_t err;
    int32_t next_pattern;  // streaming greedy: patterns handed to slots
    int32_t done_count;    // ... patterns it has finished with
    int32_t expired;       // ... the deadline passed
    int32_t idlers;        // ... warps without work
    int32_t blocks_bump, teams_bump;  // ... task blocks and teams handed out for the first time
    int32_t arrived;       // ... blocks that stay
    int32_t n_ready;       // ... tasks ready to run (about)
    unsigned long long blocks_free, teams_free;  // ... stacks of free indices (stream.cu)
    unsigned long long ready[READY_STACKS];      // ... stacks of tasks ready to run
    unsigned long long bytes_greedy;
    unsigned long long bytes_mni;
    unsigned long long alg_scanned;   // greedy search: driver-slice entries scanned (A)
    unsigned long long alg_bound;     // greedy search: sum over bound partial maps of their length
    unsigned long long alg_map_words; // greedy search: words of the maps it wrote (n per map found)
    unsigned long long search_items;
    unsigned long long mni_items;
    unsigned long long mni_total;
    unsigned long long mni_next;
    unsigned long long t0_ns;     // device clock at the start of the evaluation (k_init)
};

struct Batch {
    DevGraphView G;
    const Plan *plans;
    int32_t P;
    int32_t Wmax;
    int32_t Wmin;
    int32_t sel_cap;
    uint32_t budget;      // per-round candidate chunks of one root search (0: unlimited)
    int32_t split_max;    // pieces per split (0: no split)
    uint32_t sid_all;     // saved sub-search indices a pattern may use (bit set)
    PatState *st;
    uint32_t *used;       // [P][words]
    int32_t *dirty;       // [P][DIRTY_CAP] words of `used` made non-zero (nullable: not tracked)
    int32_t *win_root;    // [P][2][Wmax]  two window buffers per pattern
    int32_t *win_state;   // [P][2][Wmax]
    int32_t *win_map;     // [P][2][Wmax][8] (by level)
    int2 *items;          // [P*Wmax] (pattern, buffer * Wmax + slot)
    Ctl *ctl;
    int32_t *sel;         // [P][sel_cap][8] selected maps, canonical vertex order
    unsigned long long *mni_seg;  // [P*8+1] prefix sums of MNI candidate segments
    int32_t *alist;               // [2][P] patterns still in their greedy phase (nullable: all)
    uint32_t *susp;               // [P][KSUSP][DFS_SAVE_STRIDE] saved search states
    flexis_support_result *results;
    unsigned long long deadline_ns;  // > 0: the MNI pass stops this long after ctl->t0_ns
};


// The device's global nanosecond clock (PTX special register %globaltimer).
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

constexpr int DFS_SAVE_WORDS = (int)(offsetof(WarpState, need) / 4);
constexpr int DFS_SAVE_STRIDE = 192;  // words per saved sub-search
constexpr int SUSP_STATUS = DFS_SAVE_WORDS;      // SS_* of the saved sub-search
constexpr int SUSP_NEXT = DFS_SAVE_WORDS + 1;    // next sub-search of the same slot, or -1
constexpr int SUSP_MAP = DFS_SAVE_WORDS + 2;     // its map (by level) when SS_FOUND
static_assert(SUSP_MAP + MAXN <= DFS_SAVE_STRIDE, "saved search state too large");
constexpr int KSUSP = 32;             // saved sub-searches a pattern may hold at once
constexpr uint32_t SEARCH_BUDGET = 4096;  // candidate chunks a root search runs per round

constexpr int SEARCH_THREADS = 256;
constexpr int DIRTY_CAP = 1024;  // listed used-bitmap words per pattern (4 KB)

}  // namespace fx

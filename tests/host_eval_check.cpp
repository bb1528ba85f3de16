// Host check of the evaluation driver (csrc/api.cpp) on a device that is a stand-in: how a set of patterns
// is cut into batches when the streaming greedy's buffers find no room.  The stand-in holds FREE bytes, takes
// STREAM bytes for the streaming buffers and WINDOWED a pattern for the windowed rounds, and refuses what
// does not fit.
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "fx_dev.h"

using namespace fx;

static int fails = 0;
#define CHECK(c)                                                              \
    do {                                                                      \
        if (!(c)) {                                                           \
            if (fails < 10) printf("FAIL line %d: %s\n", __LINE__, #c);       \
            fails++;                                                          \
        }                                                                     \
    } while (0)

constexpr int64_t STREAMED = 1500, WINDOWED = 200'000;  // bytes a pattern
static int64_t free_bytes = 0, stream_bytes = 0;
static int streamed_room = 0;  // streamed evaluations that find room before there is none
struct Call {
    bool streamed;
    int32_t P;
};
static std::vector<Call> calls;

namespace fx {

struct DeviceGraph {};

static int fake_eval(const Plan *plans, int32_t P, flexis_support_result *out, const EvalConfig &cfg, flexis_stats *st) {
    if (st) memset(st, 0, sizeof *st);
    if (cfg.streamed) {
        if (streamed_room-- <= 0 && stream_bytes > free_bytes) return EVAL_NO_STREAM_ROOM;
        CHECK(P * STREAMED <= free_bytes);
    } else if (P * WINDOWED > free_bytes) {
        return FLEXIS_E_NOMEM;
    }
    calls.push_back({cfg.streamed, P});
    if (st) st->total_ms = cfg.search_budget > 0 ? 1e6f / (float)cfg.search_budget : 1e6f;  // the largest budget is fastest
    for (int32_t i = 0; i < P && out; i++) {
        memset(&out[i], 0, sizeof out[i]);
        out[i].status = plans[i].status;
        out[i].sigma = plans[i].sigma;
        out[i].rounds = cfg.streamed ? 1 : 2;
    }
    return FLEXIS_OK;
}

int dev_graph_build(int64_t nv, const int32_t *labels, int64_t ne, const int32_t *src, const int32_t *dst, uint64_t seed,
                    int id_order, int, HostGraph &hg, DeviceGraph **out) {
    *out = new DeviceGraph();
    return build_host_graph(nv, labels, ne, src, dst, seed, id_order, hg, 0);
}
int dev_graph_create(const HostGraph &, int, DeviceGraph **out) { *out = new DeviceGraph(); return FLEXIS_OK; }
void dev_graph_destroy(DeviceGraph *g) { delete g; }
void dev_graph_load_info(const DeviceGraph *, int64_t *b, int32_t *d) { *b = 0; *d = 0; }
int dev_graph_layout(const DeviceGraph *, int32_t, void *, int64_t, int64_t *) { return FLEXIS_E_INVALID; }
int dev_graph_device(const DeviceGraph *) { return 0; }
int64_t dev_graph_bytes(const DeviceGraph *) { return 0; }
int dev_graph_props(const DeviceGraph *, int *sm, int *l2) { *sm = *l2 = 1; return FLEXIS_OK; }
cudaStream_t dev_graph_stream(const DeviceGraph *) { return nullptr; }
int dev_eval(DeviceGraph *, const flexis_plan *, int32_t P, flexis_support_result *, cudaStream_t, const EvalConfig &cfg,
             flexis_stats *st) {
    return fake_eval(nullptr, P, nullptr, cfg, st);
}
int dev_eval_host(DeviceGraph *, const Plan *plans, int32_t P, flexis_support_result *out, const EvalConfig &cfg,
                  flexis_stats *st) {
    return fake_eval(plans, P, out, cfg, st);
}
int dev_selected(DeviceGraph *, int32_t, int32_t *, int64_t, int64_t *) { return FLEXIS_E_INVALID; }
int dev_pattern_bytes(const DeviceGraph *, int32_t, int32_t, bool streamed, int64_t *bytes) {
    *bytes = streamed ? STREAMED : WINDOWED;
    return FLEXIS_OK;
}
int dev_support_noalloc(DeviceGraph *, const Plan *, flexis_support_result *, cudaStream_t, int32_t) { return FLEXIS_E_INVALID; }
int dev_free_bytes(const DeviceGraph *, int64_t *bytes) { *bytes = free_bytes; return FLEXIS_OK; }
int dev_overlap_read(DeviceGraph *, int32_t, int32_t *, int64_t, int64_t *, int32_t *, int64_t, int64_t *) { return FLEXIS_E_INVALID; }
int serve_create(DeviceGraph *, int32_t, int32_t, int32_t, int32_t, ServeSession **) { return FLEXIS_E_INVALID; }
void serve_destroy(ServeSession *) {}
int serve_slot_bytes(const DeviceGraph *, int32_t, int64_t *) { return FLEXIS_E_INVALID; }
int serve_cancel(ServeSession *, const int32_t *, int32_t) { return FLEXIS_E_INVALID; }
int serve_step(ServeSession *, const int32_t *, const Plan *, int32_t, int32_t *, flexis_support_result *, int32_t *) {
    return FLEXIS_E_INVALID;
}

}  // namespace fx

extern "C" {
cudaError_t cudaMemcpy2DAsync(void *dst, size_t dp, const void *src, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
    for (size_t i = 0; i < h; i++) memcpy((char *)dst + i * dp, (const char *)src + i * sp, w);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *fr, size_t *tot) { *fr = *tot = (size_t)free_bytes; return cudaSuccess; }
}

int main() {
    const int32_t labels[4] = {0, 1, 0, 1}, src[3] = {0, 1, 2}, dst[3] = {1, 2, 3};
    int32_t pl[2] = {0, 1}, pe[2] = {0, 1};
    for (int autotune = -1; autotune <= 0; autotune++)
        for (int32_t count : {1, 2, 500, 6000})
            for (int room = 0; room < 2; room++) {  // with and without room for the streaming buffers
                flexis_options opt;
                flexis_default_options(&opt);
                opt.autotune = autotune;
                flexis_graph *g = nullptr;
                free_bytes = 1 << 30;
                stream_bytes = room ? free_bytes / 2 : free_bytes + 1;
                streamed_room = 0;
                calls.clear();
                CHECK(flexis_load_graph(4, labels, 3, src, dst, &opt, &g) == FLEXIS_OK);
                std::vector<flexis_pattern> pats((size_t)count);
                std::vector<int64_t> sigma((size_t)count);
                std::vector<double> lam((size_t)count, 0.5);
                for (int32_t i = 0; i < count; i++) {
                    memset(&pats[(size_t)i], 0, sizeof(flexis_pattern));
                    pats[(size_t)i].n = 2;
                    pats[(size_t)i].m = 1;
                    pats[(size_t)i].labels = pl;
                    pats[(size_t)i].edges = pe;
                    sigma[(size_t)i] = i + 1;
                }
                std::vector<flexis_support_result> res((size_t)count);
                for (auto &r : res) r.status = 99;
                CHECK(flexis_support_batch(g, pats.data(), sigma.data(), lam.data(), count, FLEXIS_MODE_EARLY, res.data()) == FLEXIS_OK);
                for (int32_t i = 0; i < count; i++)
                    CHECK(res[(size_t)i].status == FLEXIS_OK && res[(size_t)i].sigma == i + 1 &&
                          res[(size_t)i].rounds == (room ? 1 : 2));
                int64_t windowed = 0;
                for (auto &c : calls)
                    if (!c.streamed && (c.P >= 512 || autotune < 0)) windowed = std::max<int64_t>(windowed, c.P);
                // cut to a third of the memory, and not to single patterns
                if (!room) CHECK(windowed == 0 || windowed == std::min<int64_t>(count, free_bytes / 3 / WINDOWED));
                if (room) CHECK(windowed == 0);
                // one pattern, and plans in device memory, as many as the rounds have room for
                flexis_support_result one;
                CHECK(flexis_support(g, &pats[0], 7, 0.5, FLEXIS_MODE_EARLY, &one) == FLEXIS_OK && one.sigma == 7);
                std::vector<flexis_plan> plans((size_t)count);
                std::vector<int64_t> num((size_t)count, FLEXIS_LAMBDA_DEN / 2);
                CHECK(flexis_compile(g, pats.data(), sigma.data(), num.data(), FLEXIS_LAMBDA_DEN, count, FLEXIS_MODE_EARLY,
                                     plans.data()) == FLEXIS_OK);
                calls.clear();
                const int32_t dp = std::min<int32_t>(count, (int32_t)(free_bytes / WINDOWED));
                CHECK(flexis_support_plans_device(g, plans.data(), dp, res.data(), nullptr) == FLEXIS_OK);
                CHECK(calls.size() == 1 && calls[0].P == dp && calls[0].streamed == (room == 1));
                flexis_free_graph(g);
            }
    // the room goes after the first of several streamed batches: what it gave stays, the rest is cut again
    {
        flexis_options opt;
        flexis_default_options(&opt);
        opt.autotune = -1;
        flexis_graph *g = nullptr;
        free_bytes = 256ll << 20;  // (a batch may always take 256 MB)
        stream_bytes = free_bytes + 1;
        streamed_room = 1;
        calls.clear();
        CHECK(flexis_load_graph(4, labels, 3, src, dst, &opt, &g) == FLEXIS_OK);
        const int32_t first = (int32_t)((256ll << 20) / STREAMED), count = first + 5000;
        std::vector<flexis_pattern> pats((size_t)count);
        std::vector<int64_t> sigma((size_t)count);
        std::vector<double> lam((size_t)count, 0.5);
        for (int32_t i = 0; i < count; i++) {
            memset(&pats[(size_t)i], 0, sizeof(flexis_pattern));
            pats[(size_t)i].n = 2;
            pats[(size_t)i].m = 1;
            pats[(size_t)i].labels = pl;
            pats[(size_t)i].edges = pe;
            sigma[(size_t)i] = i + 1;
        }
        std::vector<flexis_support_result> res((size_t)count);
        CHECK(flexis_support_batch(g, pats.data(), sigma.data(), lam.data(), count, FLEXIS_MODE_EARLY, res.data()) == FLEXIS_OK);
        for (int32_t i = 0; i < count; i++)
            CHECK(res[(size_t)i].sigma == i + 1 && res[(size_t)i].rounds == (i < first ? 1 : 2));
        CHECK(calls.size() > 1 && calls[0].streamed && calls[0].P == first);
        for (size_t k = 1; k < calls.size(); k++) CHECK(!calls[k].streamed);
        flexis_free_graph(g);
    }
    // a budget timed under the streaming greedy, which has none, is not the windowed rounds': those time their own
    {
        flexis_options opt;
        flexis_default_options(&opt);
        flexis_graph *g = nullptr;
        free_bytes = 4ll << 30;
        stream_bytes = 0;
        streamed_room = 0;
        CHECK(flexis_load_graph(4, labels, 3, src, dst, &opt, &g) == FLEXIS_OK);
        const int32_t count = 6000;
        flexis_pattern p;
        memset(&p, 0, sizeof p);
        p.n = 2;
        p.m = 1;
        p.labels = pl;
        p.edges = pe;
        std::vector<flexis_pattern> pats((size_t)count, p);
        std::vector<int64_t> sigma((size_t)count, 3);
        std::vector<double> lam((size_t)count, 0.5);
        std::vector<flexis_support_result> res((size_t)count);
        for (int turn = 0; turn < 3; turn++) {
            if (turn == 1) stream_bytes = free_bytes + 1;
            CHECK(flexis_support_batch(g, pats.data(), sigma.data(), lam.data(), count, FLEXIS_MODE_EARLY, res.data()) == FLEXIS_OK);
            flexis_stats st;
            CHECK(flexis_last_stats(g, &st) == FLEXIS_OK);
            CHECK(st.autotune_probes == (turn < 2 ? 3 : 0));
            CHECK(st.search_budget == (turn == 0 ? 4096 : 16384));
        }
        flexis_free_graph(g);
    }
    printf("fails %d\n", fails);
    return fails != 0;
}

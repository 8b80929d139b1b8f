// C ABI of the library (include/tc.h): graph objects, device memory and the order
// of the device phases.
//
// Device memory comes from one stream-ordered pool per device (cudaMemPool with an
// unlimited release threshold), so repeated create/destroy cycles reuse memory
// without returning it to the driver and without device-wide synchronisation.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <unordered_map>
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "tc_internal.h"

using namespace tcg;

namespace tcg {
static std::atomic<uint64_t> g_launches{0};
void count_launch(int k) { g_launches.fetch_add((uint64_t)k, std::memory_order_relaxed); }
uint64_t launch_total() { return g_launches.load(std::memory_order_relaxed); }
}  // namespace tcg

namespace {

thread_local char g_last_error[256] = "";

void set_error(const char* where, cudaError_t e) {
    snprintf(g_last_error, sizeof(g_last_error), "%s: %s", where, cudaGetErrorString(e));
}

struct DeviceState {
    bool ready = false;
    int sms = 0;
    cudaMemPool_t pool = nullptr;
};

std::mutex g_dev_mutex;
DeviceState g_dev[64];

// What a graph needs of the driver beside memory: the second stream and its events, the
// events of the build and count phases, and the copy stream and events of host input.
// Sets are handed from a destroyed graph to the next one of the device: creating them
// took 20 us per graph, and 500 us with eight threads doing so at once.  A set is handed on
// once its streams are idle, so that no graph waits for a former owner's work; events are
// recorded anew.  At most SYNC_KEEP sets stay, until tc_release_cached_graphs.
struct SyncSet {
    bool known_idle = false;  // given back by a graph that had waited for all its work: not asked (5 us)
    cudaStream_t side = nullptr, copy = nullptr;  // null: could not be created, the graph's own stream does it
    cudaEvent_t fork = nullptr, join = nullptr, landed = nullptr, allocated = nullptr;
    cudaEvent_t ev[PH_EVENTS] = {};
    cudaEvent_t bev[BP_EVENTS] = {};

    cudaError_t create() {
        cudaError_t e = cudaSuccess;
        for (cudaStream_t* s : {&side, &copy})
            if (cudaStreamCreateWithFlags(s, cudaStreamNonBlocking) != cudaSuccess) {
                *s = nullptr;
                cudaGetLastError();
            }
        for (cudaEvent_t* x : {&fork, &join, &landed, &allocated})
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(x, cudaEventDisableTiming);
        for (cudaEvent_t& x : ev)
            if (e == cudaSuccess) e = cudaEventCreate(&x);
        for (cudaEvent_t& x : bev)
            if (e == cudaSuccess) e = cudaEventCreate(&x);
        return e;
    }
    // Queries are refused while any thread captures in global mode, unless relaxed for the call.
    bool idle() const {
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        cudaThreadExchangeStreamCaptureMode(&mode);
        const bool yes = cudaStreamQuery(side) == cudaSuccess && cudaStreamQuery(copy) == cudaSuccess;
        cudaThreadExchangeStreamCaptureMode(&mode);
        if (!yes) cudaGetLastError();  // cudaErrorNotReady
        return yes;
    }
    void destroy() {
        for (cudaEvent_t x : {fork, join, landed, allocated})
            if (x) cudaEventDestroy(x);
        for (cudaEvent_t x : ev)
            if (x) cudaEventDestroy(x);
        for (cudaEvent_t x : bev)
            if (x) cudaEventDestroy(x);
        for (cudaStream_t x : {side, copy})
            if (x) cudaStreamDestroy(x);
        *this = SyncSet{};
    }
};
constexpr size_t SYNC_KEEP = 64, SYNC_LOOK = 4;
std::mutex g_sync_mutex;
std::vector<SyncSet> g_sync[64];  // per device

cudaError_t take_sync(int dev, SyncSet* out) {
    {
        std::lock_guard<std::mutex> lock(g_sync_mutex);
        std::vector<SyncSet>& kept = g_sync[dev];
        // the ones given back first are the likeliest to be idle
        for (size_t k = 0; k < kept.size() && k < SYNC_LOOK; ++k) {
            if (!kept[k].known_idle && !kept[k].idle()) continue;
            *out = kept[k];
            kept.erase(kept.begin() + (std::ptrdiff_t)k);
            return cudaSuccess;
        }
    }
    const cudaError_t e = out->create();
    if (e != cudaSuccess) out->destroy();
    return e;
}

void give_sync(int dev, SyncSet* s) {
    {
        std::lock_guard<std::mutex> lock(g_sync_mutex);
        if (g_sync[dev].size() < SYNC_KEEP && s->side && s->copy) {
            try {
                g_sync[dev].push_back(*s);
                *s = SyncSet{};
                return;
            } catch (const std::bad_alloc&) {
            }
        }
    }
    s->destroy();
}

tc_status init_device(int dev, DeviceState** out) {
    if (dev < 0 || dev >= 64) return TC_ECUDA;
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    DeviceState& D = g_dev[dev];
    if (!D.ready) {
        cudaError_t e = cudaDeviceGetAttribute(&D.sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) {
            set_error("cudaDeviceGetAttribute", e);
            return TC_ECUDA;
        }
        cudaMemPoolProps props;
        memset(&props, 0, sizeof(props));
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        e = cudaMemPoolCreate(&D.pool, &props);
        if (e != cudaSuccess) {
            set_error("cudaMemPoolCreate", e);
            return TC_ECUDA;
        }
        uint64_t thr = UINT64_MAX;
        cudaMemPoolSetAttribute(D.pool, cudaMemPoolAttrReleaseThreshold, &thr);
        if ((e = build_init_attributes()) != cudaSuccess || (e = intersect_init_attributes()) != cudaSuccess) {
            set_error("cudaFuncSetAttribute", e);
            return TC_ECUDA;
        }
        D.ready = true;
    }
    *out = &D;
    return TC_OK;
}

}  // namespace

namespace tcg {
void set_last_error(const char* where, cudaError_t e) { set_error(where, e); }

cudaMemPool_t device_pool(int dev) {
    DeviceState* D = nullptr;
    return init_device(dev, &D) == TC_OK ? D->pool : nullptr;
}
}  // namespace tcg

struct tc_graph {
    int device = 0;
    cudaStream_t stream = nullptr;
    cudaMemPool_t pool = nullptr;
    Launch L{};
    int32_t n = 0;
    int64_t m_in = 0;
    int64_t m_alloc = 0;  // capacity of col / in-edge arrays
    int32_t* rank = nullptr;
    int64_t* rowstart = nullptr;
    int32_t* rowlen = nullptr;
    int2* rowinfo = nullptr;
    int32_t* col = nullptr;
    int32_t* deg = nullptr;
    int32_t* small_list[4] = {nullptr, nullptr, nullptr, nullptr};
    int32_t* cta_list = nullptr;
    int32_t hub_cap = 0;
    uint32_t* hub_cnt = nullptr;
    int64_t* hub_start = nullptr;
    unsigned long long* hub_cur64 = nullptr;
    int32_t* big_list = nullptr;
    int32_t* long_list = nullptr;
    int4* win_task = nullptr;
    int4* low_task = nullptr;
    uint2* winrow = nullptr;
    uint4* winlow = nullptr;
    uint4* win = nullptr;
    uint2* in_rec = nullptr;
    int32_t* rowof = nullptr;
    void* plan_tmp = nullptr;
    int64_t dplus_bound = 0;          // no N+(u) has more entries
    int32_t src_lo = 0, src_hi = -1;  // ranks of the sources counted (-1: up to n); tc_count_shard
    int32_t core_cap = 0;
    int32_t core_words = 0;
    uint32_t* core_bits = nullptr;  // adjacency rows; core in-degrees, lowest, highest neighbour, highest out-neighbour

    unsigned long long* t_rank = nullptr;
    DevStats* stats = nullptr;
    std::vector<void*> blocks;
    bool planned = false;
    bool counted = false;
    mutable bool verified = false;  // the statistics have been read since the last build, plan or count, without a flag
    bool plan_zeroed = false;   // the planner's part of the statistics is zero
    bool count_zeroed = false;  // t and the count's part of the statistics are zero
    Strategy strat{};
    bool timed = false;
    bool build_timed = false;
    // batch of graphs counted as one disjoint union (tc_batch_create)
    int32_t batch_G = -1;
    int32_t* batch_vbase = nullptr;   // device, G + 1
    int* batch_err = nullptr;         // device flag of the relabel and the per-graph reduction
    bool ranked_by_graph = false;     // ranks run graph by graph
    int64_t hub_reach_m = 0;          // pairs of the graphs that have vertices among the last hub_cap
    bool capture = false;             // work is being recorded into a CUDA graph: no events
    // streams and events (not while recording a CUDA graph); the second stream runs the
    // long rows' sort and the plan's hub part (single graphs only)
    SyncSet sync;
    bool has_sync = false;
    mutable bool side_busy = false;   // the second stream may hold work
    bool side_joined = true;          // the graph's stream waits for that work
    bool plan_forked = false;         // the last plan ran its hub part on the second stream
};

namespace {

tc_status cuda_fail(const char* where, cudaError_t e) {
    set_error(where, e);
    return TC_ECUDA;
}

#define TC_CK(call)                                                 \
    do {                                                            \
        cudaError_t e_ = (call);                                    \
        if (e_ != cudaSuccess) return cuda_fail(#call, e_);         \
    } while (0)

template <typename T>
tc_status dalloc(tc_graph* g, T** p, size_t count, std::vector<void*>* track) {
    size_t bytes = count * sizeof(T);
    if (bytes == 0) bytes = 16;
    bytes = (bytes + 255) & ~(size_t)255;
    void* q = nullptr;
    // while recording a CUDA graph the allocation becomes a graph memory node
    cudaError_t e = g->capture ? cudaMallocAsync(&q, bytes, g->stream)
                               : cudaMallocFromPoolAsync(&q, bytes, g->pool, g->stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("cudaMallocFromPoolAsync", e);
        return TC_ENOMEM;
    }
    track->push_back(q);
    *p = static_cast<T*>(q);
    return TC_OK;
}

// Arrays of one allocation: listed with add, placed by alloc (each on a 256-byte
// boundary).  A graph's forty arrays took 60 us to allocate and free one by one.
class Slab {
  public:
    template <typename T>
    Slab& add(T** p, size_t count) {
        items_.push_back({[](void* at, void* field) { *static_cast<T**>(field) = static_cast<T*>(at); }, p, bytes_});
        bytes_ += (count * sizeof(T) + 255) & ~(size_t)255;
        return *this;
    }
    // Room of at least `bytes` from `from` on (an earlier end), for a second use of the arrays there.
    void reach(size_t from, size_t bytes) { bytes_ = std::max(bytes_, (from + bytes + 255) & ~(size_t)255); }
    size_t end() const { return bytes_; }
    tc_status alloc(tc_graph* g, std::vector<void*>* track) {
        char* base = nullptr;
        const tc_status st = dalloc(g, &base, bytes_, track);
        if (st != TC_OK) return st;
        for (const Item& i : items_) i.set(base + i.offset, i.field);
        return TC_OK;
    }

  private:
    struct Item {
        void (*set)(void* at, void* field);
        void* field;
        size_t offset;
    };
    std::vector<Item> items_;
    size_t bytes_ = 0;
};

void free_list(tc_graph* g, std::vector<void*>* list) {
    for (void* p : *list) cudaFreeAsync(p, g->stream);
    list->clear();
}

tc_status new_graph(int32_t n, void* stream, tc_graph** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail("cudaGetDevice", e);
    DeviceState* D = nullptr;
    tc_status st = init_device(dev, &D);
    if (st != TC_OK) return st;
    tc_graph* g = new (std::nothrow) tc_graph();
    if (!g) return TC_ENOMEM;
    g->device = dev;
    g->stream = static_cast<cudaStream_t>(stream);
    g->pool = D->pool;
    g->L.stream = g->stream;
    g->L.sms = D->sms;
    g->n = n;
    for (int b = 0; b < TC_NUM_BUCKETS; ++b) {
        g->strat.strat[b] = TC_STRAT_AUTO;
        g->strat.factor[b] = 1.0f;
    }
    g->strat.strat[TC_BUCKET_SMALL] = TC_STRAT_HASH;
    g->strat.strat[TC_BUCKET_CTA] = TC_STRAT_BITMAP;
    g->strat.hub_min_degree = HUB_MIN_DEGREE;
    g->strat.hub_max = HUB_BM_BITS;
    g->strat.hub_big_in = 128;
    g->strat.hub_core = CORE_MAX;
    *out = g;
    return TC_OK;
}

tc_status read_stats(const tc_graph* g, DevStats* h) {
    TC_CK(cudaMemcpyAsync(h, g->stats, sizeof(DevStats), cudaMemcpyDeviceToHost, g->stream));
    TC_CK(cudaStreamSynchronize(g->stream));
    if (g->side_joined) g->side_busy = false;
    return TC_OK;
}

// The statistics of a built graph.  A guard of the build, the plan or the count that has
// fired (rows that could not be filled are empty) fails every call that answers from the
// graph.
tc_status read_result_stats(const tc_graph* g, DevStats* h) {
    const tc_status st = read_stats(g, h);
    if (st != TC_OK) return st;
    if (h->err & ERR_OVERFLOW) {
        snprintf(g_last_error, sizeof(g_last_error), "internal count mismatch (overflow guard)");
        return TC_EINTERNAL;
    }
    g->verified = true;
    return TC_OK;
}

// The same check for calls that wait for the stream but need no statistics.
tc_status verify(const tc_graph* g) {
    if (g->verified) return TC_OK;
    DevStats h;
    return read_result_stats(g, &h);
}

// Pairs from which rows are filled by buckets.  Whole calls, direct fill / buckets, uniform
// and R-MAT graphs: 200,000 pairs 0.28 / 0.29 and 0.36 / 0.35 ms; 1 M 0.34 / 0.35 and
// 0.54 / 0.50; 4 M 0.75 / 0.73 and 0.95 / 0.90; 32 M 2.65 / 2.18 and 5.30 / 5.08.
constexpr int64_t BUCKET_MIN_M = (int64_t)1 << 20;

int64_t isqrt(int64_t x) {  // floor of the square root
    int64_t r = (int64_t)std::sqrt((double)x);
    while (r > 0 && r * r > x) --r;
    while ((r + 1) * (r + 1) <= x) ++r;
    return r;
}

int bits_for(unsigned x) {
    int b = 0;
    while (b < 32 && (x >> b) != 0) ++b;
    return b;
}

// Builds the oriented CSR from device-resident pairs (src, dst) of length m.
// checked: read the id check back before continuing (one stream synchronisation)
// so that create can fail with TC_EINVAL; otherwise the build never waits on the
// device (the radix sort takes its degree bits from the bound 2m) and invalid ids
// are reported by the first call that reads the statistics.
// Host input of build_graph: the pairs are copied in INGEST_PIECES pieces on a side
// stream and each piece's degree counts start as soon as it has landed, so the copy
// overlaps the ingest pass.
struct HostPairs {
    const int32_t* src;
    const int32_t* dst;
    cudaStream_t side;
    cudaEvent_t landed;
};
constexpr int INGEST_PIECES = 8;

// Batches: the graphs' union id offsets and the widths of the rank key fields.
struct SegInfo {
    const int32_t* vbase;  // device, G + 1
    int32_t G;
    int seg_bits, deg_bits, local_bits;
    int64_t m_max;        // pairs of the largest graph
    int64_t hub_reach_m;  // pairs of the graphs that hubs can reach
};

// The graph's streams and events, taken at first use.
tc_status need_sync(tc_graph* g) {
    if (g->has_sync) return TC_OK;
    const cudaError_t e = take_sync(g->device, &g->sync);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return cuda_fail("streams and events", e);
    }
    g->has_sync = true;
    return TC_OK;
}

// The second stream, for single graphs that are not recorded into a CUDA graph.
const PlanStreams* side_streams(tc_graph* g, PlanStreams* out) {
    if (g->capture || g->batch_G >= 0 || !g->has_sync || !g->sync.side) return nullptr;
    *out = PlanStreams{g->sync.side, g->sync.fork, g->sync.join};
    return out;
}

tc_status build_graph(tc_graph* g, const int32_t* src, const int32_t* dst, int64_t m, bool checked = true,
                      const HostPairs* host = nullptr, const SegInfo* seg = nullptr, bool dir_bits = false,
                      bool rows_only = false) {
    const int32_t n = g->n;
    const size_t nn = (size_t)n;
    tc_status st;
    std::vector<void*>& keep = g->blocks;
    g->m_alloc = m;
    g->hub_cap = n < HUB_BM_BITS ? n : HUB_BM_BITS;
    const size_t hc = (size_t)g->hub_cap;
    g->core_cap = g->hub_cap < CORE_MAX ? g->hub_cap : CORE_MAX;
    g->core_words = core_words_for(g->core_cap);
    const size_t cc = (size_t)g->core_cap;
    if (!g->capture && (st = need_sync(g)) != TC_OK) return st;
    // rows may be filled by buckets: room for two slots per pair
    const bool buckets = seg ? m > 0 : m >= BUCKET_MIN_M;
    BuildBuffers B{};
    Slab kept, work;
    kept.add(&g->stats, 1).add(&g->t_rank, nn).add(&g->rank, nn).add(&g->rowstart, nn + 1).add(&g->rowlen, nn).add(&g->rowinfo, nn);
    kept.add(&g->col, (size_t)m).add(&g->deg, nn);
    // the zeroed counters first: one memset
    work.add(&B.dmulti, nn).add(&B.dupin, nn).add(&B.rowcnt, nn + 1).add(&B.bcount, (size_t)BUCKET_MAX + 1);
    work.add(&B.bcap, (size_t)BUCKET_MAX).add(&B.bstart, (size_t)BUCKET_MAX + 1).add(&B.bfirst, (size_t)BUCKET_MAX + 1);
    // The arrays of the plan serve the build for its pairs, rank keys and row lists first.  So
    // the peak beside the input is 92 n + 4 m + max(16 m, 12 m + 16 win_vec_cap) bytes and
    // arrays of a fixed size, never above 40 m + 100 n.  Rows alone need the build's part only.
    Slab& plan = rows_only ? work : kept;
    for (int k = 0; k < 4; ++k) plan.add(&g->small_list[k], (size_t)push_list_cap(n, m, k));
    if (!rows_only) {
        kept.add(&g->cta_list, (size_t)push_list_cap(n, m, 4));
        kept.add(&g->hub_cnt, hc + 1).add(&g->hub_start, hc + 1).add(&g->hub_cur64, hc + 1).add(&g->big_list, hc + 1);
        kept.add(&g->long_list, hc + 1).add(&g->win_task, (size_t)hub_task_cap(g->hub_cap, m));
        kept.add(&g->low_task, (size_t)hub_task_cap(g->hub_cap, m)).add(&g->winrow, nn);
        kept.add((char**)&g->plan_tmp, scan_tmp_bytes((int64_t)hc + 1));
        kept.add(&g->core_bits, cc * (size_t)g->core_words + 4 * cc);
    }
    const size_t keys_at = plan.end();
    plan.add(&B.keys, 0);
    if (!rows_only) kept.add(&g->winlow, nn);
    const size_t keys_alt = (nn + 31) & ~(size_t)31;  // whole sectors
    plan.reach(keys_at, sizeof(uint64_t) * (keys_alt + nn));
    const size_t pairs_at = plan.end();
    plan.add(&B.pairs, 0);
    if (!rows_only) kept.add(&g->in_rec, (size_t)m).add(&g->rowof, (size_t)m).add(&g->win, (size_t)win_vec_cap(n, m));
    plan.reach(pairs_at, (buckets ? 2 : 1) * sizeof(int2) * (size_t)m);
    if ((st = kept.alloc(g, &keep)) != TC_OK) return st;
    std::vector<void*> scratch;
    B.src = src;
    B.dst = dst;
    B.m = m;
    B.dir_bits = dir_bits;
    B.n = n;
    if (seg) {
        // graph by graph ranks keep every graph's rows together, so the bucket fill's
        // buckets hold whole graphs and stay balanced whatever the degrees
        B.bucket_fill = m > 0;
        B.seg_vbase = seg->vbase;
        B.seg_count = seg->G;
        B.seg_bits = seg->seg_bits;
        B.seg_deg_bits = seg->deg_bits;
        B.local_bits = seg->local_bits;
        g->hub_reach_m = seg->hub_reach_m;
        g->ranked_by_graph = seg->G > 0 && seg->seg_bits + seg->deg_bits + seg->local_bits <= 64;
    }
    size_t tmp_bytes = scan_tmp_bytes((int64_t)nn + 1);
    size_t rt = radix_tmp_bytes((int64_t)nn);
    if (rt > tmp_bytes) tmp_bytes = rt;
    char* tmp = nullptr;
    work.add(&tmp, tmp_bytes);
    if ((st = work.alloc(g, &scratch)) != TC_OK) return st;
    const size_t zeroed = (size_t)((char*)B.bcap - (char*)B.dmulti);
    B.seg = reinterpret_cast<uint32_t*>(g->deg);  // free until the rows are sorted
    B.keys_alt = B.keys + keys_alt;
    B.tmp = tmp;
    B.oriented = B.pairs;  // one or the other
    B.longlist = g->small_list[0];
    B.midlist = g->small_list[1];
    B.midlist2 = g->small_list[2];
    B.rank = g->rank;
    B.rowstart = g->rowstart;
    B.rowlen = g->rowlen;
    B.rowinfo = g->rowinfo;
    B.col = g->col;
    B.deg = g->deg;
    B.stats = g->stats;
    cudaEvent_t* const bev = g->capture ? nullptr : g->sync.bev;
    if (bev) cudaEventRecord(bev[BP_START], g->stream);
    // the statistics and t (for the first count), then the build's counters
    cudaMemsetAsync(g->stats, 0, (size_t)((char*)(g->t_rank + nn) - (char*)g->stats), g->stream);
    cudaMemsetAsync(B.dmulti, 0, zeroed, g->stream);
    g->count_zeroed = g->plan_zeroed = true;
    if (host && m > 0) {
        const int64_t piece = (m + INGEST_PIECES - 1) / INGEST_PIECES;
        cudaError_t e = cudaSuccess;
        for (int64_t first = 0; first < m && e == cudaSuccess; first += piece) {
            const int64_t cnt = first + piece < m ? piece : m - first;
            e = cudaMemcpyAsync(const_cast<int32_t*>(src) + first, host->src + first, sizeof(int32_t) * (size_t)cnt,
                                cudaMemcpyHostToDevice, host->side);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(const_cast<int32_t*>(dst) + first, host->dst + first,
                                    sizeof(int32_t) * (size_t)cnt, cudaMemcpyHostToDevice, host->side);
            if (e == cudaSuccess) e = cudaEventRecord(host->landed, host->side);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(g->stream, host->landed, 0);
            if (e == cudaSuccess) launch_canon_degree_part(B, first, cnt, g->L);
        }
        if (e != cudaSuccess) {
            free_list(g, &scratch);
            return cuda_fail("host input copy", e);
        }
        launch_max_deg(B, g->L);
    } else {
        launch_canon_degree(B, g->L);
    }
    if (bev) cudaEventRecord(bev[BP_INGEST], g->stream);
    // The vertices of N+(u) all have at least u's own pairs, of which there are at least
    // |N+(u)|, so |N+(u)|^2 <= 2 m (of its own graph, in a batch).
    B.row_bound = m;
    g->dplus_bound = isqrt(2 * (seg ? seg->m_max : m));
    int deg_bits = bits_for((unsigned)(2 * m < (int64_t)UINT32_MAX ? 2 * m : (int64_t)UINT32_MAX));
    if (checked) {
        DevStats h;
        if ((st = read_stats(g, &h)) != TC_OK) {
            free_list(g, &scratch);
            return st;
        }
        if (h.err & ERR_BAD_ID) {
            free_list(g, &scratch);
            snprintf(g_last_error, sizeof(g_last_error), "vertex id outside [0, n)");
            return TC_EINVAL;
        }
        deg_bits = bits_for(h.max_deg);
        B.row_bound = h.max_deg;
        if (g->dplus_bound > (int64_t)h.max_deg) g->dplus_bound = h.max_deg;
        // Rows through buckets, even ones for flat degrees (the largest within 64x the mean).  A
        // flat graph with one heavy vertex takes the skewed ones too, which are then filled
        // unevenly: 1 M vertices and 8.7 M pairs, 4.2 M and 44 M, whole calls by even / skewed
        // buckets / direct fill 1.02 / 1.05 / 1.05 and 7.18 / 7.45 / 8.19 ms.
        const double mean = n > 0 ? 2.0 * (double)m / (double)n : 0.0;
        B.skewed = (double)h.max_deg > 64.0 * mean;
        B.bucket_fill = m >= BUCKET_MIN_M && (!B.skewed || skewed_buckets_fit(n));
    }
    launch_rank(B, deg_bits, g->L);
    if (bev) cudaEventRecord(bev[BP_RANK], g->stream);
    PlanStreams psv{};
    g->side_busy = true;  // joined by launch_orient
    launch_orient(B, g->L, bev, seg ? nullptr : side_streams(g, &psv));
    if (bev) {
        cudaEventRecord(bev[BP_END], g->stream);
        g->build_timed = n > 0;  // else no phase has run, and its events may be a former graph's
    }
    free_list(g, &scratch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail("build kernels", e);
    return TC_OK;
}

// The highest ranks of a batch, its hubs, are vertices of its last graphs, and the plan and
// the count of the hub part walk all of it (0.47 of 10.1 ms for 66 M pairs in 840 graphs of
// which the hubs reach 16).  Where the graphs that hubs can reach have less than an eighth
// of the pairs they are left out, unless the caller has set them.
constexpr int64_t BATCH_HUB_SHARE = 8;

CountBuffers count_buffers(tc_graph* g) {
    CountBuffers C{};
    C.n = g->n;
    C.rowstart = g->rowstart;
    C.rowlen = g->rowlen;
    C.rowinfo = g->rowinfo;
    C.col = g->col;
    C.deg = g->deg;
    for (int i = 0; i < 4; ++i) C.small_list[i] = g->small_list[i];
    C.cta_list = g->cta_list;
    C.hub_cap = g->hub_cap;
    C.hub_cnt = g->hub_cnt;
    C.hub_start = g->hub_start;
    C.hub_cur64 = g->hub_cur64;
    C.big_list = g->big_list;
    C.long_list = g->long_list;
    C.win_task = g->win_task;
    C.low_task = g->low_task;
    C.winrow = g->winrow;
    C.winlow = g->winlow;
    C.win = g->win;
    C.win_cap = win_vec_cap(g->n, g->m_alloc);
    C.in_rec = g->in_rec;
    C.rowof = g->rowof;
    C.m_cap = g->m_alloc;
    C.tmp = g->plan_tmp;
    C.core_cap = g->core_cap;
    C.core_words = g->core_words;
    const size_t rows = (size_t)g->core_cap * (size_t)g->core_words;
    C.core_z = g->core_bits;
    C.core_cnt = g->core_bits + rows;
    C.core_lo = reinterpret_cast<int32_t*>(C.core_cnt + g->core_cap);
    C.core_hi = C.core_lo + g->core_cap;
    C.core_hiout = C.core_hi + g->core_cap;
    C.t_rank = g->t_rank;
    C.stats = g->stats;
    C.dplus_bound = g->dplus_bound;
    C.no_hubs = g->ranked_by_graph && g->hub_reach_m < g->m_in / BATCH_HUB_SHARE &&
                g->strat.hub_min_degree == HUB_MIN_DEGREE && g->strat.hub_max == HUB_BM_BITS;
    C.src_lo = g->src_lo;
    C.src_hi = g->src_hi < 0 ? g->n : g->src_hi;
    C.hub_ready = g->plan_forked ? g->sync.join : nullptr;
    return C;
}

// Orders the main stream after the hub part of the last plan (no-op when it ran on
// the main stream): before a replan, before the graph's memory is released, and
// wherever the hub lists are read outside the count.
void join_plan(tc_graph* g) {
    if (g->plan_forked) cudaStreamWaitEvent(g->stream, g->sync.join, 0);
    g->side_joined = true;
}

// Planning (a4): bucket lists and hub in-edge lists; rerun when hub settings change.
tc_status run_plan(tc_graph* g) {
    if (g->planned) return TC_OK;
    join_plan(g);  // a previous plan's hub part writes the buffers this one rewrites
    const size_t off = offsetof(DevStats, small_count), end = offsetof(DevStats, cta_next);
    if (!g->plan_zeroed) TC_CK(cudaMemsetAsync(reinterpret_cast<char*>(g->stats) + off, 0, end - off, g->stream));
    g->plan_zeroed = false;
    if (!g->capture) TC_CK(cudaEventRecord(g->sync.ev[PH_PLAN], g->stream));
    // single graphs build their hub lists on a second stream while the push buckets
    // are counted; batches (which may be recorded into a CUDA graph) keep one stream
    PlanStreams psv{};
    g->side_busy = true;
    g->side_joined = false;
    g->plan_forked = launch_plan(count_buffers(g), g->strat, g->L, side_streams(g, &psv));
    TC_CK(cudaGetLastError());
    g->planned = true;
    g->counted = false;
    g->verified = false;
    return TC_OK;
}

// t and the count's part of the statistics start at zero, which they are after the build.
tc_status zero_counts(tc_graph* g) {
    if (!g->count_zeroed) {
        const size_t off = offsetof(DevStats, cta_next);
        TC_CK(cudaMemsetAsync(g->t_rank, 0, sizeof(unsigned long long) * (size_t)g->n, g->stream));
        TC_CK(cudaMemsetAsync(reinterpret_cast<char*>(g->stats) + off, 0, sizeof(DevStats) - off, g->stream));
    }
    g->count_zeroed = false;
    return TC_OK;
}

tc_status run_count(tc_graph* g) {
    if (g->counted) return TC_OK;
    tc_status st;
    if (g->planned) {
        if (!g->capture) TC_CK(cudaEventRecord(g->sync.ev[PH_PLAN], g->stream));  // planning already done: empty phase
    } else if ((st = run_plan(g)) != TC_OK) {
        return st;
    }
    if ((st = zero_counts(g)) != TC_OK) return st;
    CountBuffers C = count_buffers(g);
    launch_intersect(C, g->strat, g->capture ? nullptr : g->sync.ev, g->L);
    g->side_joined = true;  // by C.hub_ready
    launch_sum_t(C, g->L);
    TC_CK(cudaGetLastError());
    g->counted = true;
    g->verified = false;
    g->timed = !g->capture && g->n > 0;
    return TC_OK;
}

void destroy(tc_graph* g) {
    if (!g) return;
    join_plan(g);
    free_list(g, &g->blocks);
    g->sync.known_idle = !g->side_busy;
    if (g->has_sync) give_sync(g->device, &g->sync);
    delete g;
}

tc_status finish_create(tc_graph* g, tc_status st, tc_graph** out) {
    if (st != TC_OK) {
        destroy(g);
        *out = nullptr;
        return st;
    }
    *out = g;
    return TC_OK;
}

}  // namespace

namespace tcg {

tc_status build_undirected_rows(int32_t n, int64_t m, const int32_t* src, const int32_t* dst, cudaStream_t stream,
                                bool dir_bits, tc_graph** g, UndirectedRows* out) {
    *g = nullptr;
    if (n < 0 || (dir_bits && n > (1 << 29)) || m < 0 || m > INT_MAX || (m > 0 && (!src || !dst))) return TC_EINVAL;
    tc_graph* built = nullptr;
    tc_status st = new_graph(n, stream, &built);
    if (st != TC_OK) return st;
    built->m_in = m;
    st = finish_create(built, build_graph(built, src, dst, m, true, nullptr, nullptr, dir_bits, true), g);
    if (st != TC_OK) return st;
    DevStats h;
    if ((st = read_result_stats(*g, &h)) != TC_OK) return st;
    out->m_simple = (int64_t)h.m_simple;
    out->loops = (int64_t)h.loops;
    out->rank = (*g)->rank;
    out->rowinfo = (*g)->rowinfo;
    out->rowlen = (*g)->rowlen;
    out->col = (*g)->col;
    return TC_OK;
}

}  // namespace tcg

extern "C" {

tc_status tc_graph_create_from_edges(int32_t n, int64_t m, const int32_t* src, const int32_t* dst,
                                     int mem_kind, void* cuda_stream, tc_graph** out) {
    if (!out) return TC_EINVAL;
    *out = nullptr;
    if (n < 0 || m < 0 || m > INT_MAX || (m > 0 && (!src || !dst)) ||
        (mem_kind != TC_MEM_HOST && mem_kind != TC_MEM_DEVICE))
        return TC_EINVAL;
    tc_graph* g = nullptr;
    tc_status st = new_graph(n, cuda_stream, &g);
    if (st != TC_OK) return st;
    g->m_in = m;
    if (mem_kind == TC_MEM_DEVICE) return finish_create(g, build_graph(g, src, dst, m), out);
    std::vector<void*> tmp;
    int32_t *ds = nullptr, *dd = nullptr;
    if ((st = dalloc(g, &ds, (size_t)m, &tmp)) || (st = dalloc(g, &dd, (size_t)m, &tmp))) {
        free_list(g, &tmp);
        return finish_create(g, st, out);
    }
    if ((st = need_sync(g)) != TC_OK) {
        free_list(g, &tmp);
        return finish_create(g, st, out);
    }
    // the copy stream may only touch ds and dd once their allocation is ordered
    const HostPairs hp{src, dst, g->sync.copy ? g->sync.copy : g->stream, g->sync.landed};
    cudaError_t e = cudaEventRecord(g->sync.allocated, g->stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(hp.side, g->sync.allocated, 0);
    if (e != cudaSuccess)
        st = cuda_fail("host input stream", e);
    else
        st = build_graph(g, ds, dd, m, true, &hp);
    // the build read its statistics back on g->stream, which waited for every piece:
    // the copies are complete
    if (st != TC_OK) cudaStreamSynchronize(hp.side);
    free_list(g, &tmp);
    return finish_create(g, st, out);
}

tc_status tc_graph_create_from_csr(int32_t n, const int64_t* offsets, const int32_t* adj, int mem_kind,
                                   void* cuda_stream, tc_graph** out) {
    if (!out) return TC_EINVAL;
    *out = nullptr;
    if (n < 0 || !offsets || (mem_kind != TC_MEM_HOST && mem_kind != TC_MEM_DEVICE)) return TC_EINVAL;
    int64_t m = 0;
    if (mem_kind == TC_MEM_HOST) {
        if (offsets[0] != 0) return TC_EINVAL;
        for (int32_t i = 0; i < n; ++i)
            if (offsets[i + 1] < offsets[i]) return TC_EINVAL;
        m = offsets[n];
        if (m > INT_MAX) return TC_EINVAL;
        if (m > 0 && !adj) return TC_EINVAL;
    }
    tc_graph* g = nullptr;
    tc_status st = new_graph(n, cuda_stream, &g);
    if (st != TC_OK) return st;
    std::vector<void*> tmp;
    const int64_t* doff = offsets;
    const int32_t* dadj = adj;
    DevStats* dstat = nullptr;
    if ((st = dalloc(g, &dstat, 1, &tmp))) {
        free_list(g, &tmp);
        return finish_create(g, st, out);
    }
    cudaMemsetAsync(dstat, 0, sizeof(DevStats), g->stream);
    if (mem_kind == TC_MEM_HOST) {
        int64_t* o = nullptr;
        int32_t* a = nullptr;
        if ((st = dalloc(g, &o, (size_t)n + 1, &tmp)) || (st = dalloc(g, &a, (size_t)m, &tmp))) {
            free_list(g, &tmp);
            return finish_create(g, st, out);
        }
        cudaMemcpyAsync(o, offsets, sizeof(int64_t) * ((size_t)n + 1), cudaMemcpyHostToDevice, g->stream);
        if (m > 0) cudaMemcpyAsync(a, adj, sizeof(int32_t) * (size_t)m, cudaMemcpyHostToDevice, g->stream);
        doff = o;
        dadj = a;
    } else {
        launch_check_offsets(doff, n, INT_MAX, dstat, g->L);
        DevStats h;
        int64_t last = 0;
        cudaError_t e = cudaMemcpyAsync(&h, dstat, sizeof(DevStats), cudaMemcpyDeviceToHost, g->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&last, doff + n, sizeof(int64_t), cudaMemcpyDeviceToHost, g->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
        if (e != cudaSuccess) {
            free_list(g, &tmp);
            return finish_create(g, cuda_fail("offsets check", e), out);
        }
        if (h.err || (last > 0 && !adj)) {
            free_list(g, &tmp);
            return finish_create(g, TC_EINVAL, out);
        }
        m = last;
    }
    int32_t* rows = nullptr;
    if ((st = dalloc(g, &rows, (size_t)m, &tmp))) {
        free_list(g, &tmp);
        return finish_create(g, st, out);
    }
    launch_expand_csr(doff, n, rows, dstat, g->L);
    g->m_in = m;
    st = build_graph(g, rows, dadj, m);
    free_list(g, &tmp);
    return finish_create(g, st, out);
}

tc_status tc_count(tc_graph* g, uint64_t* T_out) {
    if (!g || !T_out) return TC_EINVAL;
    tc_status st = run_count(g);
    if (st != TC_OK) return st;
    DevStats h;
    if ((st = read_result_stats(g, &h)) != TC_OK) return st;
    if (h.sum_t % 3 != 0) {
        snprintf(g_last_error, sizeof(g_last_error), "sum of t is not a multiple of 3");
        return TC_EINTERNAL;
    }
    *T_out = h.sum_t / 3;
    return TC_OK;
}

tc_status lcc_compute(tc_graph* g, uint64_t* t_out, double* lcc_out, int mem_kind) {
    if (!g || (mem_kind != TC_MEM_HOST && mem_kind != TC_MEM_DEVICE)) return TC_EINVAL;
    tc_status st = run_count(g);
    if (st != TC_OK) return st;
    if (!t_out && !lcc_out) return TC_OK;
    if (mem_kind == TC_MEM_DEVICE) {
        launch_finalize(g->n, g->rank, g->t_rank, g->deg, reinterpret_cast<unsigned long long*>(t_out), lcc_out,
                        g->L);
        TC_CK(cudaGetLastError());
        return TC_OK;
    }
    std::vector<void*> tmp;
    unsigned long long* dt = nullptr;
    double* dl = nullptr;
    if ((t_out && (st = dalloc(g, &dt, (size_t)g->n, &tmp))) || (lcc_out && (st = dalloc(g, &dl, (size_t)g->n, &tmp)))) {
        free_list(g, &tmp);
        return st;
    }
    launch_finalize(g->n, g->rank, g->t_rank, g->deg, dt, dl, g->L);
    cudaError_t e = cudaSuccess;
    if (t_out && g->n > 0)
        e = cudaMemcpyAsync(t_out, dt, sizeof(uint64_t) * (size_t)g->n, cudaMemcpyDeviceToHost, g->stream);
    if (e == cudaSuccess && lcc_out && g->n > 0)
        e = cudaMemcpyAsync(lcc_out, dl, sizeof(double) * (size_t)g->n, cudaMemcpyDeviceToHost, g->stream);
    free_list(g, &tmp);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
    if (e != cudaSuccess) return cuda_fail("lcc_compute copy", e);
    return verify(g);
}

// Counts one shard, then restores the whole source range on every path out (the
// next count plans again).
struct ShardRange {
    tc_graph* g;
    ShardRange(tc_graph* g_, int32_t lo, int32_t hi) : g(g_) { set(lo, hi); }
    ~ShardRange() { set(0, -1); }
    void set(int32_t lo, int32_t hi) {
        g->src_lo = lo;
        g->src_hi = hi;
        g->planned = false;
        g->counted = false;
    }
};

tc_status tc_count_shard(tc_graph* g, int32_t shard, int32_t nshards, uint64_t* t_out, int mem_kind,
                         uint64_t* T_out) {
    if (!g || nshards < 1 || shard < 0 || shard >= nshards) return TC_EINVAL;
    if (t_out && mem_kind != TC_MEM_HOST && mem_kind != TC_MEM_DEVICE) return TC_EINVAL;
    const int32_t n = g->n;
    int32_t hb[2] = {0, n};
    if (nshards > 1 && n > 0) {
        std::vector<void*> tmp;
        uint32_t* cost = nullptr;
        int64_t* prefix = nullptr;
        int32_t* bounds = nullptr;
        char* stmp = nullptr;
        tc_status st;
        if ((st = dalloc(g, &cost, (size_t)n, &tmp)) || (st = dalloc(g, &prefix, (size_t)n + 1, &tmp)) ||
            (st = dalloc(g, &bounds, 2, &tmp)) || (st = dalloc(g, &stmp, scan_tmp_bytes((int64_t)n), &tmp))) {
            free_list(g, &tmp);
            return st;
        }
        launch_shard_bounds(n, g->rowlen, cost, prefix, stmp, shard, nshards, bounds, g->L);
        cudaError_t e = cudaMemcpyAsync(hb, bounds, sizeof(hb), cudaMemcpyDeviceToHost, g->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
        free_list(g, &tmp);
        if (e != cudaSuccess) return cuda_fail("shard bounds", e);
        if (hb[0] < 0 || hb[1] < hb[0] || hb[1] > n) return TC_EINTERNAL;
    }
    ShardRange range(g, hb[0], hb[1]);
    tc_status st = run_count(g);
    if (st != TC_OK) return st;
    DevStats h;
    if ((st = read_result_stats(g, &h)) != TC_OK) return st;
    if (h.sum_t % 3 != 0) {
        snprintf(g_last_error, sizeof(g_last_error), "internal count mismatch in a shard");
        return TC_EINTERNAL;
    }
    if (T_out) *T_out = h.sum_t / 3;
    if (!t_out || n == 0) return TC_OK;
    if (mem_kind == TC_MEM_DEVICE) {
        launch_finalize(n, g->rank, g->t_rank, g->deg, reinterpret_cast<unsigned long long*>(t_out), nullptr, g->L);
        TC_CK(cudaGetLastError());
        return TC_OK;
    }
    std::vector<void*> tmp;
    unsigned long long* dt = nullptr;
    if ((st = dalloc(g, &dt, (size_t)n, &tmp))) return st;
    launch_finalize(n, g->rank, g->t_rank, g->deg, dt, nullptr, g->L);
    cudaError_t e = cudaMemcpyAsync(t_out, dt, sizeof(uint64_t) * (size_t)n, cudaMemcpyDeviceToHost, g->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
    free_list(g, &tmp);
    if (e != cudaSuccess) return cuda_fail("count_shard copy", e);
    return TC_OK;
}

tc_status tc_lcc_from_counts(tc_graph* g, const uint64_t* t, double* lcc_out, int mem_kind) {
    if (!g || !t || !lcc_out || (mem_kind != TC_MEM_HOST && mem_kind != TC_MEM_DEVICE)) return TC_EINVAL;
    const int32_t n = g->n;
    if (n == 0) return TC_OK;
    const unsigned long long* tt = reinterpret_cast<const unsigned long long*>(t);
    if (mem_kind == TC_MEM_DEVICE) {
        launch_lcc_from_counts(n, g->rank, g->deg, tt, lcc_out, g->L);
        TC_CK(cudaGetLastError());
        return TC_OK;
    }
    std::vector<void*> tmp;
    unsigned long long* dt = nullptr;
    double* dl = nullptr;
    tc_status st;
    if ((st = dalloc(g, &dt, (size_t)n, &tmp)) || (st = dalloc(g, &dl, (size_t)n, &tmp))) {
        free_list(g, &tmp);
        return st;
    }
    cudaError_t e = cudaMemcpyAsync(dt, t, sizeof(uint64_t) * (size_t)n, cudaMemcpyHostToDevice, g->stream);
    if (e == cudaSuccess) {
        launch_lcc_from_counts(n, g->rank, g->deg, dt, dl, g->L);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(lcc_out, dl, sizeof(double) * (size_t)n, cudaMemcpyDeviceToHost, g->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
    free_list(g, &tmp);
    if (e != cudaSuccess) return cuda_fail("lcc_from_counts", e);
    return verify(g);
}

// Scratch of the symmetric rows (tc_vertex.cu) for g; pool memory tracked in tmp.
static tc_status symmetric_buffers(tc_graph* g, const DevStats& h, VertexFormulaBuffers* V, std::vector<void*>* tmp) {
    const size_t nn = (size_t)g->n;
    *V = VertexFormulaBuffers{};
    V->n = g->n;
    V->m = (int64_t)h.m_simple;
    V->m_cap = g->m_alloc;
    V->rowstart = g->rowstart;
    V->rowlen = g->rowlen;
    V->rowinfo = g->rowinfo;
    V->col = g->col;
    V->deg = g->deg;
    char* radix_tmp = nullptr;
    char* scan_tmp = nullptr;
    unsigned* cs = nullptr;
    tc_status st;
    if ((st = dalloc(g, &V->indeg, nn, tmp)) || (st = dalloc(g, &V->sym_start, nn + 1, tmp)) ||
        (st = dalloc(g, &V->instart, nn + 1, tmp)) || (st = dalloc(g, &V->sym, (size_t)(2 * V->m), tmp)) ||
        (st = dalloc(g, &V->keys, (size_t)V->m_cap, tmp)) || (st = dalloc(g, &V->keys_alt, (size_t)V->m_cap, tmp)) ||
        (st = dalloc(g, &radix_tmp, radix_tmp_bytes(V->m_cap), tmp)) ||
        (st = dalloc(g, &scan_tmp, scan_tmp_bytes((int64_t)nn + 1), tmp)) || (st = dalloc(g, &V->t, nn, tmp)) ||
        (st = dalloc(g, &cs, 8, tmp)))
        return st;
    V->radix_tmp = radix_tmp;
    V->tmp = scan_tmp;
    V->counter = cs;
    V->sum = reinterpret_cast<unsigned long long*>(cs + 2);
    return TC_OK;
}

tc_status tc_count_vertex_formula(tc_graph* g, uint64_t* t_out, int mem_kind, uint64_t* T_out) {
    if (!g || !t_out || (mem_kind != TC_MEM_HOST && mem_kind != TC_MEM_DEVICE)) return TC_EINVAL;
    DevStats h;
    tc_status st = read_result_stats(g, &h);
    if (st != TC_OK) return st;
    if (h.err & ERR_BAD_ID) return TC_EINVAL;
    const size_t nn = (size_t)g->n;
    VertexFormulaBuffers V;
    std::vector<void*> tmp;
    unsigned long long* dt = nullptr;
    if ((st = symmetric_buffers(g, h, &V, &tmp)) != TC_OK) {
        free_list(g, &tmp);
        return st;
    }
    launch_vertex_formula(V, g->L);
    unsigned long long* out = mem_kind == TC_MEM_DEVICE ? reinterpret_cast<unsigned long long*>(t_out) : nullptr;
    if (!out && (st = dalloc(g, &dt, nn, &tmp))) {
        free_list(g, &tmp);
        return st;
    }
    launch_finalize(g->n, g->rank, V.t, g->deg, out ? out : dt, nullptr, g->L);
    unsigned long long sum = 0;
    cudaError_t e = cudaMemcpyAsync(&sum, V.sum, sizeof(sum), cudaMemcpyDeviceToHost, g->stream);
    if (e == cudaSuccess && !out && nn > 0)
        e = cudaMemcpyAsync(t_out, dt, sizeof(uint64_t) * nn, cudaMemcpyDeviceToHost, g->stream);
    free_list(g, &tmp);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
    if (e != cudaSuccess) return cuda_fail("tc_count_vertex_formula", e);
    if (sum % 3 != 0) {
        snprintf(g_last_error, sizeof(g_last_error), "sum of t is not a multiple of 3");
        return TC_EINTERNAL;
    }
    if (T_out) *T_out = sum / 3;
    return TC_OK;
}

tc_status tc_edge_support(tc_graph* g, int32_t* u_out, int32_t* v_out, uint32_t* support_out, int mem_kind) {
    if (!g || !u_out || !v_out || !support_out || (mem_kind != TC_MEM_HOST && mem_kind != TC_MEM_DEVICE))
        return TC_EINVAL;
    DevStats h;
    tc_status st = read_result_stats(g, &h);
    if (st != TC_OK) return st;
    if (h.err & ERR_BAD_ID) return TC_EINVAL;
    const size_t nn = (size_t)g->n, me = (size_t)h.m_simple;
    // the oriented count with every triangle added to its three edges instead of its
    // vertices (the dense core counts its edges' triangles by words of bits); the plan is
    // the count's own
    const Strategy saved = g->strat;
    Strategy S = saved;
    S.strat[TC_BUCKET_SMALL] = TC_STRAT_HASH;
    S.strat[TC_BUCKET_CTA] = TC_STRAT_BITMAP;
    S.strat[TC_BUCKET_HUB] = TC_STRAT_BITMAP;
    std::vector<void*> tmp;
    uint32_t* sup = nullptr;
    int32_t* id_of = nullptr;
    int64_t* estart = nullptr;
    char* stmp = nullptr;
    int32_t *du = nullptr, *dv = nullptr;
    uint32_t* ds = nullptr;
    const bool dev = mem_kind == TC_MEM_DEVICE;
    if ((st = dalloc(g, &sup, (size_t)g->m_alloc, &tmp)) || (st = dalloc(g, &id_of, nn, &tmp)) ||
        (st = dalloc(g, &estart, nn + 1, &tmp)) || (st = dalloc(g, &stmp, scan_tmp_bytes((int64_t)nn + 1), &tmp)) ||
        (!dev && ((st = dalloc(g, &du, me, &tmp)) || (st = dalloc(g, &dv, me, &tmp)) || (st = dalloc(g, &ds, me, &tmp))))) {
        free_list(g, &tmp);
        return st;
    }
    g->strat = S;
    g->counted = false;
    cudaError_t e = cudaMemsetAsync(sup, 0, sizeof(uint32_t) * (size_t)g->m_alloc, g->stream);
    if (e == cudaSuccess && (st = run_plan(g)) == TC_OK && (st = zero_counts(g)) == TC_OK) {
        CountBuffers C = count_buffers(g);
        C.sup = sup;
        launch_intersect(C, g->strat, nullptr, g->L);
        g->side_joined = true;  // by C.hub_ready; leaves parts of t in t_rank: the next count starts it anew
        launch_support_out(g->n, g->rank, g->rowlen, g->rowinfo, g->col, sup, id_of, estart, stmp, dev ? u_out : du,
                           dev ? v_out : dv, dev ? support_out : ds, g->L);
        e = cudaGetLastError();
    }
    g->strat = saved;
    g->counted = false;
    if (st != TC_OK) {
        free_list(g, &tmp);
        return st;
    }
    if (e == cudaSuccess && !dev && me > 0) {
        e = cudaMemcpyAsync(u_out, du, sizeof(int32_t) * me, cudaMemcpyDeviceToHost, g->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(v_out, dv, sizeof(int32_t) * me, cudaMemcpyDeviceToHost, g->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(support_out, ds, sizeof(uint32_t) * me, cudaMemcpyDeviceToHost, g->stream);
    }
    free_list(g, &tmp);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
    if (e != cudaSuccess) return cuda_fail("tc_edge_support", e);
    return read_result_stats(g, &h);
}

tc_status tc_remote_cache(tc_graph* g, int32_t parts, int32_t ncap, const uint64_t* capacity_bytes, uint64_t* hits,
                          uint64_t* hit_bytes, tc_remote_part* part_stats) {
    if (!g || parts < 1 || (g->n > 0 && parts > g->n) || (g->n == 0 && parts != 1) || ncap < 0 ||
        (ncap > 0 && !capacity_bytes))
        return TC_EINVAL;
    for (int32_t c = 1; c < ncap; ++c)
        if (capacity_bytes[c] < capacity_bytes[c - 1]) return TC_EINVAL;
    DevStats h;
    tc_status st = read_result_stats(g, &h);
    if (st != TC_OK) return st;
    if (h.err & ERR_BAD_ID) return TC_EINVAL;
    const size_t cells = (size_t)TC_CACHE_KINDS * (size_t)parts * (size_t)ncap;
    const size_t half = cells / 2;  // per policy: 2 caches x processes x capacities
    if (hits) memset(hits, 0, sizeof(uint64_t) * cells);
    if (hit_bytes) memset(hit_bytes, 0, sizeof(uint64_t) * cells);
    if (part_stats) memset(part_stats, 0, sizeof(tc_remote_part) * (size_t)parts);
    const int64_t ms = (int64_t)h.m_simple;
    if (g->n == 0 || ms == 0) return TC_OK;
    const size_t nn = (size_t)g->n;
    RemoteCacheBuffers R{};
    R.n = g->n;
    R.parts = parts;
    R.ncap = ncap;
    R.ms2 = 2 * ms;
    R.rank = g->rank;
    R.rowstart = g->rowstart;
    R.rowlen = g->rowlen;
    R.col = g->col;
    R.deg = g->deg;
    const int64_t big = R.ms2 > (int64_t)nn ? R.ms2 : (int64_t)nn;
    std::vector<void*> tmp;
    char *rtmp = nullptr, *stmp = nullptr;
    uint64_t* dcaps = nullptr;
    if ((st = dalloc(g, &R.id_of, nn, &tmp)) || (st = dalloc(g, &R.sdeg, nn, &tmp)) ||
        (st = dalloc(g, &R.prank, nn, &tmp)) || (st = dalloc(g, &R.vkeys, nn, &tmp)) ||
        (st = dalloc(g, &R.vkeys_alt, nn, &tmp)) || (st = dalloc(g, &R.estart, nn + 1, &tmp)) ||
        (st = dalloc(g, &R.keys, (size_t)R.ms2, &tmp)) || (st = dalloc(g, &R.keys_alt, (size_t)R.ms2, &tmp)) ||
        (st = dalloc(g, &R.flag, (size_t)R.ms2, &tmp)) || (st = dalloc(g, &R.pos, (size_t)R.ms2 + 1, &tmp)) ||
        (st = dalloc(g, &R.item, (size_t)R.ms2, &tmp)) || (st = dalloc(g, &R.part, (size_t)R.ms2, &tmp)) ||
        (st = dalloc(g, &R.pc, (size_t)parts, &tmp)) || (st = dalloc(g, &rtmp, radix_tmp_bytes(big), &tmp)) ||
        (st = dalloc(g, &stmp, scan_tmp_bytes(big + 1), &tmp)) || (st = dalloc(g, &dcaps, (size_t)ncap, &tmp)) ||
        (st = dalloc(g, &R.cnt, half, &tmp)) || (st = dalloc(g, &R.byt, half, &tmp)) ||
        (st = dalloc(g, &R.sc_cnt, half, &tmp)) || (st = dalloc(g, &R.sc_byt, half, &tmp))) {
        free_list(g, &tmp);
        return st;
    }
    R.radix_tmp = rtmp;
    R.scan_tmp = stmp;
    R.caps = dcaps;
    cudaError_t e = cudaSuccess;
    if (ncap > 0) e = cudaMemcpyAsync(dcaps, capacity_bytes, sizeof(uint64_t) * (size_t)ncap, cudaMemcpyHostToDevice,
                                      g->stream);
    cudaMemsetAsync(R.pc, 0, sizeof(PartCounters) * (size_t)parts, g->stream);
    cudaMemsetAsync(R.cnt, 0, sizeof(unsigned long long) * half, g->stream);
    cudaMemsetAsync(R.byt, 0, sizeof(unsigned long long) * half, g->stream);
    cudaMemsetAsync(R.sc_cnt, 0, sizeof(unsigned long long) * half, g->stream);
    cudaMemsetAsync(R.sc_byt, 0, sizeof(unsigned long long) * half, g->stream);
    launch_rc_stream(R, g->L);
    uint32_t N32 = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&N32, R.pos + R.ms2, sizeof(uint32_t), cudaMemcpyDeviceToHost, g->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
    if (e != cudaSuccess) {
        free_list(g, &tmp);
        return cuda_fail("tc_remote_cache: reads", e);
    }
    const int64_t N = (int64_t)N32;
    if (N > 0) {
        const size_t n1 = (size_t)N;
        if ((st = dalloc(g, &R.prev, n1, &tmp)) || (st = dalloc(g, &R.pstart, (size_t)parts + 1, &tmp)) ||
            (st = dalloc(g, &R.key_lru, n1, &tmp)) || (st = dalloc(g, &R.wdeg, n1, &tmp)) ||
            (st = dalloc(g, &R.q_lru, n1, &tmp)) || (st = dalloc(g, &R.th_lru, n1, &tmp)) ||
            (st = dalloc(g, &R.e0deg, n1 + 1, &tmp)) ||
            (st = dalloc(g, &R.lk, (size_t)rc_levels(N) * n1, &tmp)) ||
            (st = dalloc(g, &R.le, (size_t)rc_levels(N) * (n1 + 1), &tmp)) || (st = dalloc(g, &R.la[0], n1, &tmp)) ||
            (st = dalloc(g, &R.la[1], n1, &tmp)) || (st = dalloc(g, &R.f_lru_deg, n1, &tmp)) ||
            (st = dalloc(g, &R.f_lru_one, n1, &tmp)) || (st = dalloc(g, &R.ukeys, n1, &tmp)) ||
            (st = dalloc(g, &R.udeg, n1, &tmp)) || (st = dalloc(g, &R.ubase, (size_t)parts + 1, &tmp)) ||
            (st = dalloc(g, &R.lr, n1, &tmp))) {
            free_list(g, &tmp);
            return st;
        }
        launch_rc_caches(R, N, g->L);
        // the score simulations size their bitmaps by the largest process's count of
        // distinct entries
        std::vector<int64_t> ub((size_t)parts + 1);
        e = cudaMemcpyAsync(ub.data(), R.ubase, sizeof(int64_t) * ub.size(), cudaMemcpyDeviceToHost, g->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
        if (e != cudaSuccess) {
            free_list(g, &tmp);
            return cuda_fail("tc_remote_cache: distinct entries", e);
        }
        int64_t dmax = 0;
        for (int32_t k = 0; k < parts; ++k) dmax = std::max(dmax, ub[(size_t)k + 1] - ub[(size_t)k]);
        const RcSimShape S = rc_sim_shape(dmax);
        if (!S.shared && (st = dalloc(g, &R.sim_state, S.bytes / 4 * half, &tmp))) {
            free_list(g, &tmp);
            return st;
        }
        launch_rc_score(R, S, g->L);
    }
    std::vector<unsigned long long> hc(half), hb(half), sc(half), sb(half);
    std::vector<PartCounters> hp((size_t)parts);
    e = cudaGetLastError();
    const size_t hbytes = sizeof(unsigned long long) * half;
    if (e == cudaSuccess && half) e = cudaMemcpyAsync(hc.data(), R.cnt, hbytes, cudaMemcpyDeviceToHost, g->stream);
    if (e == cudaSuccess && half) e = cudaMemcpyAsync(hb.data(), R.byt, hbytes, cudaMemcpyDeviceToHost, g->stream);
    if (e == cudaSuccess && half) e = cudaMemcpyAsync(sc.data(), R.sc_cnt, hbytes, cudaMemcpyDeviceToHost, g->stream);
    if (e == cudaSuccess && half) e = cudaMemcpyAsync(sb.data(), R.sc_byt, hbytes, cudaMemcpyDeviceToHost, g->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(hp.data(), R.pc, sizeof(PartCounters) * (size_t)parts, cudaMemcpyDeviceToHost, g->stream);
    free_list(g, &tmp);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
    if (e != cudaSuccess) return cuda_fail("tc_remote_cache", e);
    for (size_t i = 0; i < half; ++i)
        if (sc[i] == RC_SIM_BROKEN) {
            snprintf(g_last_error, sizeof(g_last_error), "tc_remote_cache: a score simulation found no entry to evict");
            return TC_EINTERNAL;
        }
    // rows of the policy arrays: cache 0 = adjacency lists, 1 = offsets
    const int lru_kind[2] = {TC_CACHE_ADJ_LRU, TC_CACHE_OFF_LRU};
    const int score_kind[2] = {TC_CACHE_ADJ_SCORE, TC_CACHE_OFF_SCORE};
    for (int w = 0; ncap > 0 && w < 2; ++w)
        for (int32_t k = 0; k < parts; ++k) {
            const size_t src = ((size_t)w * (size_t)parts + (size_t)k) * (size_t)ncap;
            const size_t dl = ((size_t)lru_kind[w] * (size_t)parts + (size_t)k) * (size_t)ncap;
            const size_t ds = ((size_t)score_kind[w] * (size_t)parts + (size_t)k) * (size_t)ncap;
            // LRU: a read that fits capacity c fits every larger one, so its hits are
            // prefix sums of the histogram; the score caches are simulated per capacity
            uint64_t cs = 0, bs = 0;
            for (int32_t c = 0; c < ncap; ++c) {
                cs += hc[src + (size_t)c];
                bs += hb[src + (size_t)c];
                if (hits) {
                    hits[dl + (size_t)c] = cs;
                    hits[ds + (size_t)c] = sc[src + (size_t)c];
                }
                if (hit_bytes) {
                    hit_bytes[dl + (size_t)c] = bs;
                    hit_bytes[ds + (size_t)c] = sb[src + (size_t)c];
                }
            }
        }
    if (part_stats)
        for (int32_t k = 0; k < parts; ++k) {
            part_stats[k].reads = (int64_t)hp[(size_t)k].reads;
            part_stats[k].top_reads = (int64_t)hp[(size_t)k].top_reads;
            part_stats[k].distinct = (int64_t)hp[(size_t)k].distinct;
            part_stats[k].read_bytes = (int64_t)hp[(size_t)k].read_bytes;
        }
    return TC_OK;
}

tc_status tc_graph_info(const tc_graph* g, int64_t* m_simple, int64_t* loops_dropped, int64_t* dups_dropped) {
    if (!g) return TC_EINVAL;
    DevStats h;
    tc_status st = read_result_stats(g, &h);
    if (st != TC_OK) return st;
    if (m_simple) *m_simple = (int64_t)h.m_simple;
    if (loops_dropped) *loops_dropped = (int64_t)h.loops;
    if (dups_dropped) *dups_dropped = g->m_in - (int64_t)h.loops - (int64_t)h.m_simple;
    return TC_OK;
}

tc_status tc_graph_size(const tc_graph* g, int32_t* n, int64_t* m_oriented) {
    if (!g) return TC_EINVAL;
    if (n) *n = g->n;
    if (m_oriented) {
        DevStats h;
        tc_status st = read_result_stats(g, &h);
        if (st != TC_OK) return st;
        *m_oriented = (int64_t)h.m_simple;
    }
    return TC_OK;
}

void tc_graph_destroy(tc_graph* g) { destroy(g); }

const char* tc_status_str(tc_status s) {
    switch (s) {
        case TC_OK: return "TC_OK: success";
        case TC_EINVAL: return "TC_EINVAL: invalid argument";
        case TC_ENOMEM: return "TC_ENOMEM: out of memory";
        case TC_ECUDA: return "TC_ECUDA: CUDA runtime error";
        case TC_ETIMEOUT: return "TC_ETIMEOUT: device-side wait timed out";
        case TC_EBUSY: return "TC_EBUSY: resource busy";
        case TC_EINTERNAL: return "TC_EINTERNAL: internal consistency check failed";
    }
    return "unknown tc_status";
}

const char* tc_last_error_detail(void) { return g_last_error; }

tc_status tc_graph_set_strategy(tc_graph* g, int bucket, int strategy, double factor) {
    if (!g || bucket < 0 || bucket >= TC_NUM_BUCKETS || strategy < TC_STRAT_AUTO || strategy > TC_STRAT_HASH ||
        !(factor > 0.0))
        return TC_EINVAL;
    if (bucket == TC_BUCKET_SMALL && (strategy == TC_STRAT_PROBE || strategy == TC_STRAT_BITMAP)) return TC_EINVAL;
    if (bucket != TC_BUCKET_SMALL && strategy == TC_STRAT_HASH) return TC_EINVAL;
    if (bucket == TC_BUCKET_HUB && (strategy == TC_STRAT_MERGE || strategy == TC_STRAT_SEARCH)) return TC_EINVAL;
    g->strat.strat[bucket] = strategy;
    g->strat.factor[bucket] = (float)factor;
    g->counted = false;
    return TC_OK;
}

tc_status tc_graph_set_hubs(tc_graph* g, int32_t min_degree, int32_t max_hubs) {
    if (!g || min_degree < 0 || max_hubs < 0) return TC_EINVAL;
    g->strat.hub_min_degree = min_degree;
    g->strat.hub_max = max_hubs < HUB_BM_BITS ? max_hubs : HUB_BM_BITS;
    g->planned = false;
    g->counted = false;
    return TC_OK;
}

tc_status tc_graph_build_timing(const tc_graph* g, float* ms, int count) {
    if (!g || !ms || count < 0 || !g->build_timed) return TC_EINVAL;
    TC_CK(cudaEventSynchronize(g->sync.bev[BP_END]));
    float v[BP_EVENTS] = {};
    for (int i = 1; i < BP_EVENTS; ++i) TC_CK(cudaEventElapsedTime(&v[i - 1], g->sync.bev[i - 1], g->sync.bev[i]));
    TC_CK(cudaEventElapsedTime(&v[BP_EVENTS - 1], g->sync.bev[BP_START], g->sync.bev[BP_END]));
    for (int i = 0; i < count && i < BP_EVENTS; ++i) ms[i] = v[i];
    return TC_OK;
}

tc_status tc_graph_last_timing(const tc_graph* g, float* ms, int count) {
    if (!g || !ms || count < 0) return TC_EINVAL;
    if (!g->timed) return TC_EINVAL;
    TC_CK(cudaEventSynchronize(g->sync.ev[PH_END]));
    float v[5] = {0, 0, 0, 0, 0};
    TC_CK(cudaEventElapsedTime(&v[0], g->sync.ev[PH_PLAN], g->sync.ev[PH_SMALL]));
    TC_CK(cudaEventElapsedTime(&v[1], g->sync.ev[PH_SMALL], g->sync.ev[PH_CTA]));
    TC_CK(cudaEventElapsedTime(&v[2], g->sync.ev[PH_CTA], g->sync.ev[PH_HUB]));
    TC_CK(cudaEventElapsedTime(&v[3], g->sync.ev[PH_HUB], g->sync.ev[PH_END]));
    TC_CK(cudaEventElapsedTime(&v[4], g->sync.ev[PH_PLAN], g->sync.ev[PH_END]));
    for (int i = 0; i < count && i < 5; ++i) ms[i] = v[i];
    return TC_OK;
}

tc_status tc_graph_plan_stats(tc_graph* g, int64_t* edges, int64_t* ids) {
    if (!g || !edges || !ids) return TC_EINVAL;
    tc_status st = run_plan(g);
    if (st != TC_OK) return st;
    join_plan(g);
    const int nb = TC_NUM_BUCKETS + 1;
    unsigned long long* d = nullptr;
    TC_CK(cudaMallocFromPoolAsync((void**)&d, sizeof(unsigned long long) * 2 * nb, g->pool, g->stream));
    unsigned long long h[2 * (TC_NUM_BUCKETS + 1)] = {};
    cudaMemsetAsync(d, 0, sizeof(h), g->stream);
    launch_plan_stats(count_buffers(g), d, g->L);
    cudaError_t e = cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, g->stream);
    cudaFreeAsync(d, g->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
    if (e != cudaSuccess) return cuda_fail("tc_graph_plan_stats", e);
    for (int b = 0; b < nb; ++b) {
        edges[b] = (int64_t)h[b];
        ids[b] = (int64_t)h[nb + b];
    }
    return TC_OK;
}

uint64_t tc_launch_count(void) { return launch_total(); }

// ---- batches ------------------------------------------------------------------

static tc_status batch_host_checks(int32_t G, const int32_t* n, const int64_t* edge_off, int64_t* n_total,
                                   int64_t* m) {
    if (G < 0 || (G > 0 && (!n || !edge_off))) return TC_EINVAL;
    int64_t tot = 0;
    if (G > 0 && edge_off[0] != 0) return TC_EINVAL;
    for (int32_t g = 0; g < G; ++g) {
        if (n[g] < 0 || edge_off[g + 1] < edge_off[g]) return TC_EINVAL;
        tot += n[g];
    }
    if (tot > INT_MAX) return TC_EINVAL;
    *n_total = tot;
    *m = G > 0 ? edge_off[G] : 0;
    if (*m > INT_MAX) return TC_EINVAL;
    return TC_OK;
}

// Device pipeline of a batch (no host synchronisation: capturable).
// Widths of the (graph, degree, local id) rank key of a batch, from the host arrays:
// a vertex's pair count is at most its graph's pair count.
static SegInfo batch_seg_info(int32_t G, const int32_t* n, const int64_t* edge_off, const int32_t* vbase_dev) {
    SegInfo s{vbase_dev, G, 1, 1, 1, 0, 0};
    int32_t nmax = 1;
    int64_t mmax = 1;
    for (int32_t i = 0; i < G; ++i) {
        if (n[i] > nmax) nmax = n[i];
        if (edge_off[i + 1] - edge_off[i] > mmax) mmax = edge_off[i + 1] - edge_off[i];
    }
    s.m_max = mmax;
    int64_t reached = 0;
    for (int32_t i = G - 1; i >= 0 && reached < HUB_BM_BITS; --i) {
        reached += n[i];
        s.hub_reach_m += edge_off[i + 1] - edge_off[i];
    }
    while (s.seg_bits < 31 && ((int64_t)1 << s.seg_bits) < (int64_t)G) ++s.seg_bits;
    while (s.local_bits < 31 && ((int64_t)1 << s.local_bits) < (int64_t)nmax) ++s.local_bits;
    while (s.deg_bits < 33 && ((int64_t)1 << s.deg_bits) <= mmax) ++s.deg_bits;
    return s;
}

static tc_status batch_build(tc_graph* g, int32_t G, const int32_t* vbase_dev, const int64_t* eoff_dev,
                             const int32_t* src, const int32_t* dst, int64_t m, const SegInfo* seg) {
    std::vector<void*> tmp;
    int32_t *us = nullptr, *ud = nullptr;
    tc_status st;
    if ((st = dalloc(g, &us, (size_t)m, &tmp)) || (st = dalloc(g, &ud, (size_t)m, &tmp))) {
        free_list(g, &tmp);
        return st;
    }
    launch_batch_relabel(G, eoff_dev, vbase_dev, src, dst, m, us, ud, g->batch_err, g->L);
    st = build_graph(g, us, ud, m, false, nullptr, seg);
    free_list(g, &tmp);
    return st;
}

extern "C" tc_status tc_batch_create(int32_t G, const int32_t* n, const int64_t* edge_off, const int32_t* src,
                                     const int32_t* dst, int mem_kind, void* cuda_stream, tc_graph** out) {
    if (!out) return TC_EINVAL;
    *out = nullptr;
    int64_t n_total = 0, m = 0;
    tc_status st = batch_host_checks(G, n, edge_off, &n_total, &m);
    if (st != TC_OK) return st;
    if ((m > 0 && (!src || !dst)) || (mem_kind != TC_MEM_HOST && mem_kind != TC_MEM_DEVICE)) return TC_EINVAL;
    tc_graph* g = nullptr;
    if ((st = new_graph((int32_t)n_total, cuda_stream, &g)) != TC_OK) return st;
    g->m_in = m;
    g->batch_G = G;
    std::vector<int32_t> vb((size_t)G + 1, 0);
    for (int32_t i = 0; i < G; ++i) vb[i + 1] = vb[i] + n[i];
    std::vector<void*> tmp;
    int64_t* eoff = nullptr;
    if ((st = dalloc(g, &g->batch_vbase, (size_t)G + 1, &g->blocks)) || (st = dalloc(g, &g->batch_err, 1, &g->blocks)) ||
        (st = dalloc(g, &eoff, (size_t)G + 1, &tmp)))
        return finish_create(g, st, out);
    cudaMemsetAsync(g->batch_err, 0, sizeof(int), g->stream);
    cudaError_t e = cudaMemcpyAsync(g->batch_vbase, vb.data(), sizeof(int32_t) * vb.size(), cudaMemcpyHostToDevice,
                                    g->stream);
    if (e == cudaSuccess && G > 0)
        e = cudaMemcpyAsync(eoff, edge_off, sizeof(int64_t) * ((size_t)G + 1), cudaMemcpyHostToDevice, g->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);  // host arrays may be pageable and short-lived
    if (e != cudaSuccess) {
        free_list(g, &tmp);
        return finish_create(g, cuda_fail("tc_batch_create copy", e), out);
    }
    const int32_t* s_dev = src;
    const int32_t* d_dev = dst;
    if (mem_kind == TC_MEM_HOST && m > 0) {
        int32_t *hs = nullptr, *hd = nullptr;
        if ((st = dalloc(g, &hs, (size_t)m, &tmp)) || (st = dalloc(g, &hd, (size_t)m, &tmp))) {
            free_list(g, &tmp);
            return finish_create(g, st, out);
        }
        e = cudaMemcpyAsync(hs, src, sizeof(int32_t) * (size_t)m, cudaMemcpyHostToDevice, g->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(hd, dst, sizeof(int32_t) * (size_t)m, cudaMemcpyHostToDevice, g->stream);
        if (e != cudaSuccess) {
            free_list(g, &tmp);
            return finish_create(g, cuda_fail("tc_batch_create copy", e), out);
        }
        s_dev = hs;
        d_dev = hd;
    }
    const SegInfo seg = batch_seg_info(G, n, edge_off, g->batch_vbase);
    st = batch_build(g, G, g->batch_vbase, eoff, s_dev, d_dev, m, &seg);
    free_list(g, &tmp);
    return finish_create(g, st, out);
}

static tc_status batch_count_device(tc_graph* g, unsigned long long* T_dev) {
    tc_status st = run_count(g);
    if (st != TC_OK) return st;
    launch_batch_T(g->batch_G, g->batch_vbase, g->ranked_by_graph ? nullptr : g->rank, g->t_rank, T_dev, g->batch_err, g->L);
    TC_CK(cudaGetLastError());
    return TC_OK;
}

static tc_status batch_check(tc_graph* g) {
    int err = 0;
    DevStats h;
    TC_CK(cudaMemcpyAsync(&err, g->batch_err, sizeof(int), cudaMemcpyDeviceToHost, g->stream));
    tc_status st = read_stats(g, &h);  // synchronises
    if (st != TC_OK) return st;
    if ((err | h.err) & ERR_BAD_ID) {
        snprintf(g_last_error, sizeof(g_last_error), "vertex id outside [0, n_g) in a batch graph");
        return TC_EINVAL;
    }
    if (((err | h.err) & ERR_OVERFLOW) || h.sum_t % 3 != 0) return TC_EINTERNAL;
    return TC_OK;
}

extern "C" tc_status tc_batch_count(tc_graph* g, uint64_t* T_out, int mem_kind) {
    if (!g || g->batch_G < 0 || (g->batch_G > 0 && !T_out) || (mem_kind != TC_MEM_HOST && mem_kind != TC_MEM_DEVICE))
        return TC_EINVAL;
    const int32_t G = g->batch_G;
    tc_status st;
    if (mem_kind == TC_MEM_DEVICE) {
        if ((st = batch_count_device(g, reinterpret_cast<unsigned long long*>(T_out))) != TC_OK) return st;
        return batch_check(g);
    }
    std::vector<void*> tmp;
    unsigned long long* dT = nullptr;
    if ((st = dalloc(g, &dT, (size_t)G + 1, &tmp)) != TC_OK) return st;
    if ((st = batch_count_device(g, dT)) == TC_OK) {
        cudaError_t e = G > 0 ? cudaMemcpyAsync(T_out, dT, sizeof(uint64_t) * (size_t)G, cudaMemcpyDeviceToHost, g->stream)
                              : cudaSuccess;
        if (e != cudaSuccess) st = cuda_fail("tc_batch_count copy", e);
    }
    free_list(g, &tmp);
    if (st != TC_OK) return st;
    return batch_check(g);
}

extern "C" tc_status tc_batch_size(const tc_graph* g, int32_t* G) {
    if (!g || !G || g->batch_G < 0) return TC_EINVAL;
    *G = g->batch_G;
    return TC_OK;
}

// ---- tuning and autotuner --------------------------------------------------------

static tc_status tuning_check(const tc_tuning* t) {
    if (!t) return TC_EINVAL;
    for (int b = 0; b < TC_NUM_BUCKETS; ++b) {
        const int s = t->strategy[b];
        if (s < TC_STRAT_AUTO || s > TC_STRAT_HASH || !(t->factor[b] > 0.0)) return TC_EINVAL;
        if (b == TC_BUCKET_SMALL && (s == TC_STRAT_PROBE || s == TC_STRAT_BITMAP)) return TC_EINVAL;
        if (b != TC_BUCKET_SMALL && s == TC_STRAT_HASH) return TC_EINVAL;
        if (b == TC_BUCKET_HUB && (s == TC_STRAT_MERGE || s == TC_STRAT_SEARCH)) return TC_EINVAL;
    }
    if (t->hub_min_degree < 0 || t->hub_max < 0 || t->hub_big_in < 1 || t->hub_core < 0) return TC_EINVAL;
    return TC_OK;
}

static void tuning_get(const Strategy& S, tc_tuning* t) {
    for (int b = 0; b < TC_NUM_BUCKETS; ++b) {
        t->strategy[b] = S.strat[b];
        t->factor[b] = S.factor[b];
    }
    t->hub_min_degree = S.hub_min_degree;
    t->hub_max = S.hub_max;
    t->hub_big_in = S.hub_big_in;
    t->hub_core = S.hub_core;
}

static void tuning_put(tc_graph* g, const tc_tuning* t) {
    const bool replan = g->strat.hub_min_degree != t->hub_min_degree || g->strat.hub_max != t->hub_max ||
                        g->strat.hub_big_in != t->hub_big_in || g->strat.hub_core != t->hub_core;
    for (int b = 0; b < TC_NUM_BUCKETS; ++b) {
        g->strat.strat[b] = t->strategy[b];
        g->strat.factor[b] = (float)t->factor[b];
    }
    g->strat.hub_min_degree = t->hub_min_degree;
    g->strat.hub_max = t->hub_max < HUB_BM_BITS ? t->hub_max : HUB_BM_BITS;
    g->strat.hub_big_in = t->hub_big_in;
    g->strat.hub_core = t->hub_core < CORE_MAX ? t->hub_core : CORE_MAX;
    if (replan) g->planned = false;
    g->counted = false;
}

static tc_tuning default_tuning() {
    tc_tuning t;
    for (int b = 0; b < TC_NUM_BUCKETS; ++b) {
        t.strategy[b] = TC_STRAT_AUTO;
        t.factor[b] = 1.0;
    }
    t.strategy[TC_BUCKET_SMALL] = TC_STRAT_HASH;
    t.strategy[TC_BUCKET_CTA] = TC_STRAT_BITMAP;
    t.hub_min_degree = HUB_MIN_DEGREE;
    t.hub_max = HUB_BM_BITS;
    t.hub_big_in = 128;
    t.hub_core = CORE_MAX;
    return t;
}

extern "C" tc_status tc_graph_get_tuning(const tc_graph* g, tc_tuning* out) {
    if (!g || !out) return TC_EINVAL;
    tuning_get(g->strat, out);
    return TC_OK;
}

extern "C" tc_status tc_graph_set_tuning(tc_graph* g, const tc_tuning* t) {
    if (!g) return TC_EINVAL;
    tc_status st = tuning_check(t);
    if (st != TC_OK) return st;
    tuning_put(g, t);
    return TC_OK;
}

static std::mutex g_tune_mutex;
static std::unordered_map<uint64_t, tc_tuning> g_tune_cache;

// Count once under the current settings and return the phase times (ms[0..4]).
static tc_status timed_count(tc_graph* g, float* ms) {
    g->counted = false;
    tc_status st = run_count(g);
    if (st != TC_OK) return st;
    return tc_graph_last_timing(g, ms, 5);
}

extern "C" tc_status tc_graph_autotune(tc_graph* g, int32_t force, tc_tuning* out) {
    if (!g) return TC_EINVAL;
    tc_tuning best = default_tuning();
    tuning_put(g, &best);
    int64_t e[TC_NUM_BUCKETS + 1], ids[TC_NUM_BUCKETS + 1];
    tc_status st = tc_graph_plan_stats(g, e, ids);
    if (st != TC_OK) return st;
    // signature: powers of two of the planned work per bucket and of the graph size
    uint64_t sig = 1469598103934665603ull;
    auto mix = [&](int64_t x) {
        const uint64_t q = (uint64_t)std::llround(std::log2((double)x + 1.0));
        sig = (sig ^ q) * 1099511628211ull;
    };
    mix(g->n);
    for (int b = 0; b <= TC_NUM_BUCKETS; ++b) {
        mix(e[b]);
        mix(ids[b]);
    }
    if (!force) {
        std::lock_guard<std::mutex> lock(g_tune_mutex);
        auto it = g_tune_cache.find(sig);
        if (it != g_tune_cache.end()) {
            tuning_put(g, &it->second);
            if (out) *out = it->second;
            return TC_OK;
        }
    }
    float ms[5];
    // 1. hub threshold and block/warp split, default strategies
    const int hub_cands[][2] = {{32, 128}, {16, 128}, {64, 128}, {128, 128}, {32, 64}, {32, 256}, {32, 1024}};
    float best_total = 1e30f;
    for (const auto& hc : hub_cands) {
        tc_tuning t = default_tuning();
        t.hub_min_degree = hc[0];
        t.hub_big_in = hc[1];
        tuning_put(g, &t);
        float tot = 1e30f;
        for (int r = 0; r < 2; ++r) {
            if ((st = timed_count(g, ms)) != TC_OK) return st;
            tot = std::fmin(tot, ms[4]);
        }
        if (tot < best_total) {
            best_total = tot;
            best = t;
        }
    }
    // 2. per-bucket strategy, each bucket judged by its own kernel time
    const int sm_s[] = {TC_STRAT_HASH, TC_STRAT_AUTO, TC_STRAT_AUTO, TC_STRAT_MERGE, TC_STRAT_AUTO};
    const double sm_f[] = {1.0, 4.0, 0.25, 1.0, 1.0};  // AUTO at factors 4, 1/4 and 1
    const int cta_s[] = {TC_STRAT_BITMAP, TC_STRAT_AUTO, TC_STRAT_PROBE, TC_STRAT_SEARCH, TC_STRAT_MERGE};
    const int hub_s[] = {TC_STRAT_BITMAP, TC_STRAT_PROBE, TC_STRAT_BITMAP, TC_STRAT_PROBE, TC_STRAT_BITMAP};
    float best_b[3] = {1e30f, 1e30f, 1e30f};
    tc_tuning pick = best;
    for (int i = 0; i < 5; ++i) {
        tc_tuning t = best;
        t.strategy[TC_BUCKET_SMALL] = sm_s[i];
        t.factor[TC_BUCKET_SMALL] = sm_f[i];
        t.strategy[TC_BUCKET_CTA] = cta_s[i];
        t.strategy[TC_BUCKET_HUB] = hub_s[i];
        tuning_put(g, &t);
        float b3[3] = {1e30f, 1e30f, 1e30f};
        for (int r = 0; r < 2; ++r) {
            if ((st = timed_count(g, ms)) != TC_OK) return st;
            for (int k = 0; k < 3; ++k) b3[k] = std::fmin(b3[k], ms[1 + k]);
        }
        if (b3[0] < best_b[0]) {
            best_b[0] = b3[0];
            pick.strategy[TC_BUCKET_SMALL] = sm_s[i];
            pick.factor[TC_BUCKET_SMALL] = sm_f[i];
        }
        if (b3[1] < best_b[1]) {
            best_b[1] = b3[1];
            pick.strategy[TC_BUCKET_CTA] = cta_s[i];
        }
        if (b3[2] < best_b[2]) {
            best_b[2] = b3[2];
            pick.strategy[TC_BUCKET_HUB] = hub_s[i];
        }
    }
    tuning_put(g, &pick);
    {
        std::lock_guard<std::mutex> lock(g_tune_mutex);
        g_tune_cache[sig] = pick;
    }
    if (out) *out = pick;
    return TC_OK;
}

// ---- one-call batch, optionally recorded into a CUDA graph -----------------------

struct RunEntry {
    uint64_t key = 0;
    int device = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    int32_t* vbase = nullptr;
    int64_t* eoff = nullptr;
    int* status = nullptr;
    uint64_t kernels = 0;  // kernel launches recorded in the graph
};
static std::mutex g_run_mutex;
static std::vector<RunEntry> g_runs;

static void free_run_entry(RunEntry* r) {
    if (r->exec) cudaGraphExecDestroy(r->exec);
    if (r->graph) cudaGraphDestroy(r->graph);
    cudaFree(r->vbase);
    cudaFree(r->eoff);
    cudaFree(r->status);
    *r = RunEntry{};
}

static uint64_t fnv(uint64_t h, const void* p, size_t bytes) {
    const unsigned char* c = static_cast<const unsigned char*>(p);
    for (size_t i = 0; i < bytes; ++i) h = (h ^ c[i]) * 1099511628211ull;
    return h;
}

// The device work of one batch call on g->stream (no host synchronisation).
static tc_status batch_pipeline(tc_graph* g, int32_t G, int32_t* vbase, const int64_t* eoff, const int32_t* src,
                                const int32_t* dst, int64_t m, uint64_t* T_out, uint64_t* t_out, double* lcc_out,
                                int* status, const SegInfo* seg) {
    g->batch_G = G;
    g->batch_vbase = vbase;
    tc_status st;
    if ((st = dalloc(g, &g->batch_err, 1, &g->blocks)) != TC_OK) return st;
    TC_CK(cudaMemsetAsync(g->batch_err, 0, sizeof(int), g->stream));
    if ((st = batch_build(g, G, vbase, eoff, src, dst, m, seg)) != TC_OK) return st;
    if ((st = batch_count_device(g, reinterpret_cast<unsigned long long*>(T_out))) != TC_OK) return st;
    if (t_out || lcc_out)
        launch_finalize(g->n, g->rank, g->t_rank, g->deg, reinterpret_cast<unsigned long long*>(t_out), lcc_out, g->L);
    launch_run_status(g->stats, g->batch_err, status, g->L);
    TC_CK(cudaGetLastError());
    return TC_OK;
}

extern "C" tc_status tc_batch_run(int32_t G, const int32_t* n, const int64_t* edge_off, const int32_t* src,
                                  const int32_t* dst, uint64_t* T_out, uint64_t* t_out, double* lcc_out,
                                  const tc_tuning* tuning, void* cuda_stream, int flags) {
    int64_t n_total = 0, m = 0;
    tc_status st = batch_host_checks(G, n, edge_off, &n_total, &m);
    if (st != TC_OK) return st;
    if ((m > 0 && (!src || !dst)) || (G > 0 && !T_out)) return TC_EINVAL;
    if (tuning && (st = tuning_check(tuning)) != TC_OK) return st;
    const bool graph_mode = (flags & TC_RUN_GRAPH) != 0;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    if (graph_mode && !stream) return TC_EINVAL;
    int dev = 0;
    TC_CK(cudaGetDevice(&dev));
    DeviceState* D = nullptr;
    if ((st = init_device(dev, &D)) != TC_OK) return st;
    const tc_tuning tun = tuning ? *tuning : default_tuning();
    uint64_t key = 1469598103934665603ull;
    key = fnv(key, &G, sizeof(G));
    key = fnv(key, n, sizeof(int32_t) * (size_t)G);
    key = fnv(key, edge_off, sizeof(int64_t) * ((size_t)G + 1));
    const void* ptrs[5] = {src, dst, T_out, t_out, lcc_out};
    key = fnv(key, ptrs, sizeof(ptrs));
    key = fnv(key, &tun, sizeof(tun));
    key = fnv(key, &dev, sizeof(dev));
    RunEntry* hit = nullptr;
    if (graph_mode) {
        std::lock_guard<std::mutex> lock(g_run_mutex);
        for (auto& r : g_runs)
            if (r.key == key && r.device == dev) hit = &r;
    }
    int status_h = 0;
    if (hit) {
        TC_CK(cudaGraphLaunch(hit->exec, stream));
        count_launch((int)hit->kernels);
        TC_CK(cudaMemcpyAsync(&status_h, hit->status, sizeof(int), cudaMemcpyDeviceToHost, stream));
        TC_CK(cudaStreamSynchronize(stream));
    } else {
        RunEntry ent;
        ent.key = key;
        ent.device = dev;
        std::vector<int32_t> vb((size_t)G + 1, 0);
        for (int32_t i = 0; i < G; ++i) vb[i + 1] = vb[i] + n[i];
        tc_graph* g = nullptr;
        if ((st = new_graph((int32_t)n_total, cuda_stream, &g)) != TC_OK) return st;
        if (graph_mode) {  // arrays that the recorded graph keeps
            cudaError_t e = cudaMalloc(&ent.vbase, sizeof(int32_t) * vb.size());
            if (e == cudaSuccess) e = cudaMalloc(&ent.eoff, sizeof(int64_t) * ((size_t)G + 1));
            if (e == cudaSuccess) e = cudaMalloc(&ent.status, sizeof(int));
            if (e == cudaSuccess)
                e = cudaMemcpy(ent.vbase, vb.data(), sizeof(int32_t) * vb.size(), cudaMemcpyHostToDevice);
            if (e == cudaSuccess && G > 0)
                e = cudaMemcpy(ent.eoff, edge_off, sizeof(int64_t) * ((size_t)G + 1), cudaMemcpyHostToDevice);
            if (e != cudaSuccess) {
                free_run_entry(&ent);
                destroy(g);
                return cuda_fail("tc_batch_run arrays", e);
            }
        } else {  // of this call: released with the graph object
            Slab arrays;
            arrays.add(&ent.vbase, vb.size()).add(&ent.eoff, (size_t)G + 1).add(&ent.status, 1);
            st = arrays.alloc(g, &g->blocks);
            // pageable host memory is staged before these calls return
            cudaError_t e = cudaSuccess;
            if (st == TC_OK)
                e = cudaMemcpyAsync(ent.vbase, vb.data(), sizeof(int32_t) * vb.size(), cudaMemcpyHostToDevice, stream);
            if (st == TC_OK && e == cudaSuccess && G > 0)
                e = cudaMemcpyAsync(ent.eoff, edge_off, sizeof(int64_t) * ((size_t)G + 1), cudaMemcpyHostToDevice, stream);
            if (st == TC_OK && e != cudaSuccess) st = cuda_fail("tc_batch_run copy", e);
            if (st != TC_OK) {
                destroy(g);
                return st;
            }
        }
        g->m_in = m;
        g->capture = graph_mode;
        tuning_put(g, &tun);
        cudaError_t e = graph_mode ? cudaStreamBeginCapture(stream, cudaStreamCaptureModeThreadLocal) : cudaSuccess;
        if (e != cudaSuccess) {
            free_run_entry(&ent);
            destroy(g);
            return cuda_fail("cudaStreamBeginCapture", e);
        }
        const uint64_t k0 = launch_total();
        const SegInfo seg = batch_seg_info(G, n, edge_off, ent.vbase);
        st = batch_pipeline(g, G, ent.vbase, ent.eoff, src, dst, m, T_out, t_out, lcc_out, ent.status, &seg);
        if (!graph_mode) {
            if (st == TC_OK) {
                e = cudaMemcpyAsync(&status_h, ent.status, sizeof(int), cudaMemcpyDeviceToHost, stream);
                if (e != cudaSuccess) st = cuda_fail("tc_batch_run status", e);
            }
            destroy(g);
            e = cudaStreamSynchronize(stream);
            if (st != TC_OK) return st;
            if (e != cudaSuccess) return cuda_fail("tc_batch_run", e);
        } else {
            g->batch_vbase = nullptr;  // owned by the entry
            destroy(g);
            ent.kernels = launch_total() - k0;
            e = cudaStreamEndCapture(stream, &ent.graph);
            if (st == TC_OK && e != cudaSuccess) st = cuda_fail("cudaStreamEndCapture", e);
            if (st == TC_OK && (e = cudaGraphInstantiate(&ent.exec, ent.graph, 0)) != cudaSuccess)
                st = cuda_fail("cudaGraphInstantiate", e);
            if (st == TC_OK && (e = cudaGraphLaunch(ent.exec, stream)) != cudaSuccess)
                st = cuda_fail("cudaGraphLaunch", e);
            if (st != TC_OK) {
                free_run_entry(&ent);
                return st;
            }
            TC_CK(cudaMemcpyAsync(&status_h, ent.status, sizeof(int), cudaMemcpyDeviceToHost, stream));
            TC_CK(cudaStreamSynchronize(stream));
            std::lock_guard<std::mutex> lock(g_run_mutex);
            g_runs.push_back(ent);
        }
    }
    if (status_h & ERR_BAD_ID) {
        snprintf(g_last_error, sizeof(g_last_error), "vertex id outside [0, n_g) in a batch graph");
        return TC_EINVAL;
    }
    if (status_h & ERR_OVERFLOW) return TC_EINTERNAL;
    return TC_OK;
}

extern "C" void tc_release_cached_graphs(void) {
    {
        std::lock_guard<std::mutex> lock(g_sync_mutex);
        int cur = 0;
        const bool any = cudaGetDevice(&cur) == cudaSuccess;
        for (int dev = 0; dev < 64 && any; ++dev) {
            if (g_sync[dev].empty()) continue;
            cudaSetDevice(dev);
            for (SyncSet& x : g_sync[dev]) x.destroy();
            g_sync[dev].clear();
            cudaSetDevice(cur);
        }
    }
    std::lock_guard<std::mutex> lock(g_run_mutex);
    for (auto& r : g_runs) {
        int cur = 0;
        cudaGetDevice(&cur);
        cudaSetDevice(r.device);
        free_run_entry(&r);
        cudaSetDevice(cur);
    }
    g_runs.clear();
}

}  // extern "C"

// A CUDA runtime and the kernel launchers of the library in host memory, for tests of
// tc_api.cu's host code without a GPU: device memory is the heap, a copy or a memset
// happens at once, streams and events are numbers, and a launcher writes only the
// statistics that the host code reads back.  What a test sets up and looks at is in Fake.
#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <utility>
#include <vector>

#include "tc_internal.h"

namespace {

struct Event {
    bool recorded = false;
};

struct Fake {
    // set up by the test
    int err_after_build = 0, err_after_count = 0;  // flags that the fill and the count raise
    unsigned max_deg = 0;                          // largest degree that the ingest finds
    std::map<std::string, int> fail;               // call name: fail its k-th call from now on (1: the next)
    std::set<long> busy;                           // streams that still hold work
    // seen by the test
    long created_streams = 0, live_streams = 0, live_events = 0;
    std::vector<long> plan_side;                   // second stream of every plan (0: none)
    std::map<void*, size_t> live;
    size_t bytes = 0, peak = 0;
    std::set<long> streams;
};
Fake F;
cudaError_t last_error = cudaSuccess;

cudaError_t result(const char* name) {
    const auto it = F.fail.find(name);
    if (it == F.fail.end() || --it->second != 0) return cudaSuccess;
    F.fail.erase(it);
    return last_error = cudaErrorMemoryAllocation;
}

// Sizes of full-size graphs are only booked: nothing reads or writes such arrays here.
cudaError_t take(const char* name, void** p, size_t bytes) {
    const cudaError_t e = result(name);
    if (e != cudaSuccess) return e;
    *p = malloc(std::min(bytes, (size_t)64 << 20));
    F.live[*p] = bytes;
    F.bytes += bytes;
    F.peak = std::max(F.peak, F.bytes);
    return cudaSuccess;
}
cudaError_t give(void* p) {
    const auto it = F.live.find(p);
    if (it == F.live.end()) return p ? cudaErrorInvalidValue : cudaSuccess;
    F.bytes -= it->second;
    F.live.erase(it);
    free(p);
    return cudaSuccess;
}

}  // namespace

extern "C" {

cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 8, cudaSuccess; }
cudaError_t cudaGetLastError() { return std::exchange(last_error, cudaSuccess); }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { return *p = (cudaMemPool_t)1, cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return take("malloc", p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return take("malloc", p, n); }
cudaError_t cudaMalloc(void** p, size_t n) { return take("malloc", p, n); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return give(p); }
cudaError_t cudaFree(void* p) { return give(p); }
cudaError_t cudaMemcpyAsync(void* to, const void* from, size_t n, cudaMemcpyKind, cudaStream_t) {
    const cudaError_t e = result("memcpy");
    if (e == cudaSuccess && n <= (size_t)1 << 20) memcpy(to, from, n);
    return e;
}
cudaError_t cudaMemcpy(void* to, const void* from, size_t n, cudaMemcpyKind k) {
    return cudaMemcpyAsync(to, from, n, k, nullptr);
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
    if (n <= (size_t)1 << 20 || F.live.count(p)) memset(p, v, std::min(n, (size_t)1 << 20));
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    const cudaError_t e = result("stream");
    if (e != cudaSuccess) return e;
    *s = (cudaStream_t)(100 + ++F.created_streams);
    F.streams.insert((long)*s);
    ++F.live_streams;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { return --F.live_streams, F.streams.erase((long)s), cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t s) { return F.busy.count((long)s) ? cudaErrorNotReady : cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return result("synchronize"); }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    const cudaError_t r = result("event");
    if (r != cudaSuccess) return r;
    *e = (cudaEvent_t) new Event;
    ++F.live_events;
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return --F.live_events, delete (Event*)e, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { return ((Event*)e)->recorded = true, cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
    if (!((Event*)a)->recorded || !((Event*)b)->recorded) return last_error = cudaErrorInvalidResourceHandle;
    return *ms = 1.0f, cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return *g = (cudaGraph_t)1, cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
    return *x = (cudaGraphExec_t)1, cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }

}  // extern "C"

namespace tcg {

// Scratch sizes: those of tc_prims.cu to within a few bytes.
size_t scan_tmp_bytes(int64_t count) { return (size_t)(count / 1024 + 3) * 8 + 256; }
size_t radix_tmp_bytes(int64_t count) { return (size_t)(256 * (count / 4096 + 1)) * 4 + 512; }
int core_words_for(int32_t cap) { return ((cap + 31) / 32 + 7) & ~7; }
bool skewed_buckets_fit(int32_t n) { return n <= 52000000; }
cudaError_t build_init_attributes() { return cudaSuccess; }
cudaError_t intersect_init_attributes() { return cudaSuccess; }
int rc_levels(int64_t) { return 1; }
RcSimShape rc_sim_shape(int64_t) { return {}; }

void launch_check_offsets(const int64_t*, int32_t, int64_t, DevStats*, const Launch&) {}
void launch_expand_csr(const int64_t*, int32_t, int32_t*, DevStats*, const Launch&) {}
void launch_canon_degree(const BuildBuffers& B, const Launch&) { B.stats->max_deg = F.max_deg; }
void launch_canon_degree_part(const BuildBuffers&, int64_t, int64_t, const Launch&) {}
void launch_max_deg(const BuildBuffers& B, const Launch&) { B.stats->max_deg = F.max_deg; }
void launch_rank(const BuildBuffers&, int, const Launch&) {}
void launch_orient(const BuildBuffers& B, const Launch& L, cudaEvent_t* ev, const PlanStreams*) {
    if (B.n <= 0) return;
    if (ev)
        for (int k : {BP_COUNT, BP_FILL, BP_SORT}) cudaEventRecord(ev[k], L.stream);
    B.stats->err |= F.err_after_build;
}
bool launch_plan(const CountBuffers& C, const Strategy&, const Launch&, const PlanStreams* ps) {
    if (C.n <= 0) return false;
    F.plan_side.push_back(ps ? (long)ps->side : 0);
    return ps != nullptr;
}
void launch_intersect(const CountBuffers& C, const Strategy&, cudaEvent_t* ev, const Launch& L) {
    if (C.n <= 0) return;
    if (ev)
        for (int k : {PH_SMALL, PH_CTA, PH_HUB, PH_END}) cudaEventRecord(ev[k], L.stream);
    C.stats->err |= F.err_after_count;
}
void launch_sum_t(const CountBuffers&, const Launch&) {}
void launch_finalize(int32_t, const int32_t*, const unsigned long long*, const int32_t*, unsigned long long*, double*,
                     const Launch&) {}
void launch_lcc_from_counts(int32_t, const int32_t*, const int32_t*, const unsigned long long*, double*, const Launch&) {}
void launch_shard_bounds(int32_t n, const int32_t*, uint32_t*, int64_t*, void*, int32_t, int32_t, int32_t* bounds,
                         const Launch&) {
    bounds[0] = 0;
    bounds[1] = n;
}
void launch_vertex_formula(const VertexFormulaBuffers& V, const Launch&) { *V.sum = 0; }
void launch_support_out(int32_t, const int32_t*, const int32_t*, const int2*, const int32_t*, const uint32_t*, int32_t*,
                        int64_t*, void*, int32_t*, int32_t*, uint32_t*, const Launch&) {}
void launch_plan_stats(const CountBuffers&, unsigned long long*, const Launch&) {}
void launch_rc_stream(RemoteCacheBuffers&, const Launch&) {}
void launch_rc_caches(const RemoteCacheBuffers&, int64_t, const Launch&) {}
void launch_rc_score(const RemoteCacheBuffers&, const RcSimShape&, const Launch&) {}
void launch_batch_relabel(int32_t, const int64_t*, const int32_t*, const int32_t*, const int32_t*, int64_t, int32_t*,
                          int32_t*, int*, const Launch&) {}
void launch_batch_T(int32_t, const int32_t*, const int32_t*, const unsigned long long*, unsigned long long*, int*,
                    const Launch&) {}
void launch_run_status(const DevStats* stats, const int* batch_err, int* status, const Launch&) {
    *status = stats->err | *batch_err;
}

}  // namespace tcg

// What the tests call beside the library's own entry points.
extern "C" {

void fake_reset() {
    tc_release_cached_graphs();
    F = Fake{};
}
void fake_flags(int after_build, int after_count) { F.err_after_build = after_build, F.err_after_count = after_count; }
void fake_max_deg(unsigned d) { F.max_deg = d; }
void fake_fail(const char* call, int kth) { F.fail[call] = kth; }
void fake_busy(long stream, int on) { on ? (void)F.busy.insert(stream) : (void)F.busy.erase(stream); }
long fake_plan_side(int k) { return k < (int)F.plan_side.size() ? F.plan_side[k] : -1; }
long fake_created_streams() { return F.created_streams; }
long fake_live_streams() { return F.live_streams; }
long fake_live_events() { return F.live_events; }
size_t fake_bytes() { return F.bytes; }
size_t fake_peak() { return F.peak; }
// The rows that tc_directed_lcc works on.
int fake_undirected_rows(int32_t n, int64_t m, const int32_t* src, const int32_t* dst, int dir_bits) {
    tc_graph* g = nullptr;
    tcg::UndirectedRows rows{};
    const tc_status st = tcg::build_undirected_rows(n, m, src, dst, nullptr, dir_bits != 0, &g, &rows);
    if (g) tc_graph_destroy(g);
    return st;
}

}  // extern "C"

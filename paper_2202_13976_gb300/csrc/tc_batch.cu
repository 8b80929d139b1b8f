// Batched counting: G independent graphs are counted as one disjoint union.
//
// Graph g's pairs use local ids in [0, n_g); in the union they become
// vbase[g] + id, with vbase the exclusive prefix sum of the n_g.  A disjoint union
// has no triangle across graphs, so the union's t(v) and LCC(v) are exactly the
// per-graph values and T_g is the sum of t over graph g's vertex range divided by 3.
// Counting the union with the single-graph kernels keeps every multiprocessor
// busy even when most graphs are tiny (the planner's persistent, dynamically
// scheduled bucket kernels take vertices of all graphs from one queue), instead of
// one short launch sequence per graph.
#include "tc_device.cuh"
#include "tc_internal.h"

namespace tcg {

namespace {

// Union ids; a pair with a local id outside [0, n_g) becomes a self-loop at vbase[g]
// (dropped later) and raises ERR_BAD_ID.  A warp takes RELABEL_PAIRS consecutive pairs
// whatever graphs they belong to: it finds the first one's graph by a binary search and
// its lanes step on from there.  One block per graph left the few large graphs to a
// block each: 2.0 ms for 66 M pairs in 840 graphs, now 0.21.
constexpr int RELABEL_PAIRS = 256;

__global__ void __launch_bounds__(256) k_batch_relabel(int32_t G, const int64_t* __restrict__ edge_off,
                                                       const int32_t* __restrict__ vbase,
                                                       const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                       int64_t m, int32_t* __restrict__ usrc, int32_t* __restrict__ udst,
                                                       int* __restrict__ err) {
    const int lane = lane_id();
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    int bad = 0;
    for (int64_t p0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * RELABEL_PAIRS; p0 < m;
         p0 += warps * RELABEL_PAIRS) {
        int lo = 0, hi = G;  // the last graph whose pairs start at or before p0
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (edge_off[mid] <= p0)
                lo = mid;
            else
                hi = mid;
        }
        int g = lo;
        int64_t end = edge_off[g + 1];
        int32_t b = vbase[g], ng = vbase[g + 1] - b;
#pragma unroll
        for (int k = 0; k < RELABEL_PAIRS / 32; ++k) {
            const int64_t p = p0 + k * 32 + lane;
            if (p >= m) break;
            int32_t u = src[p], v = dst[p];
            if (p >= end) {
                do ++g;
                while (p >= edge_off[g + 1]);  // ends: p < m = edge_off[G]
                end = edge_off[g + 1];
                b = vbase[g];
                ng = vbase[g + 1] - b;
            }
            if ((uint32_t)u >= (uint32_t)ng || (uint32_t)v >= (uint32_t)ng) {
                bad = 1;
                u = 0;
                v = 0;
            }
            usrc[p] = b + u;
            udst[p] = b + v;
        }
    }
    if (bad) atomicOr(err, ERR_BAD_ID);
}

// One block per graph (grid-stride): T_g = (sum of t over the graph's vertices) / 3.  Ranks
// that run graph by graph (rank null) give a graph's counts in one piece.
constexpr int BATCH_T_THREADS = 1024;

__global__ void __launch_bounds__(BATCH_T_THREADS) k_batch_T(int32_t G, const int32_t* __restrict__ vbase,
                                                             const int32_t* __restrict__ rank,
                                                             const unsigned long long* __restrict__ t_rank,
                                                             unsigned long long* __restrict__ T_out,
                                                             int* __restrict__ err) {
    __shared__ unsigned long long ws[BATCH_T_THREADS / 32];
    for (int g = blockIdx.x; g < G; g += gridDim.x) {
        unsigned long long s = 0;
        const int64_t v1 = vbase[g + 1];
        for (int64_t v0 = vbase[g] + threadIdx.x; v0 < v1; v0 += 4 * BATCH_T_THREADS) {
            unsigned long long x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int64_t v = v0 + k * BATCH_T_THREADS;
                x[k] = v < v1 ? t_rank[rank ? rank[v] : v] : 0;
            }
            s += x[0] + x[1] + x[2] + x[3];
        }
        s = warp_sum(s);
        if (lane_id() == 0) ws[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x < 32) {
            const unsigned long long tot = warp_sum(ws[threadIdx.x]);
            if (threadIdx.x == 0) {
                if (tot % 3 != 0) atomicOr(err, ERR_OVERFLOW);
                T_out[g] = tot / 3;
            }
        }
        __syncthreads();
    }
}

// Status word of a whole batch call: id errors, failed per-graph sums, sum of t not
// a multiple of 3.
__global__ void k_run_status(const DevStats* stats, const int* batch_err, int* status) {
    int s = stats->err | *batch_err;
    if (stats->sum_t % 3 != 0) s |= ERR_OVERFLOW;
    *status = s;
}

}  // namespace

void launch_run_status(const DevStats* stats, const int* batch_err, int* status, const Launch& L) {
    k_run_status<<<1, 1, 0, L.stream>>>(stats, batch_err, status);
    count_launch();
}

void launch_batch_relabel(int32_t G, const int64_t* edge_off, const int32_t* vbase, const int32_t* src,
                          const int32_t* dst, int64_t m, int32_t* usrc, int32_t* udst, int* err, const Launch& L) {
    if (G <= 0 || m <= 0) return;
    k_batch_relabel<<<grid_for(m, 8 * RELABEL_PAIRS, L.sms, 16), 256, 0, L.stream>>>(G, edge_off, vbase, src, dst, m,
                                                                                    usrc, udst, err);
    count_launch();
}

void launch_batch_T(int32_t G, const int32_t* vbase, const int32_t* rank, const unsigned long long* t_rank,
                    unsigned long long* T_out, int* err, const Launch& L) {
    if (G <= 0) return;
    k_batch_T<<<grid_for(G, 1, L.sms, 16), BATCH_T_THREADS, 0, L.stream>>>(G, vbase, rank, t_rank, T_out, err);
    count_launch();
}

}  // namespace tcg

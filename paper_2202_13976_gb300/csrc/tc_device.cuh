// Device helpers shared by the library's kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace tcg {

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned r;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(r));
    return r;
}

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

template <typename T>
__device__ __forceinline__ T warp_max(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        T w = __shfl_xor_sync(FULL, v, o);
        v = w > v ? w : v;
    }
    return v;
}

// Inclusive warp scan.
template <typename T>
__device__ __forceinline__ T warp_inclusive_scan(T v) {
    const int lane = lane_id();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T w = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += w;
    }
    return v;
}

// Appends `want` (per lane) to a global list with one atomic per warp; returns the
// lane's slot (valid only where want is true).  All 32 lanes must call it.
__device__ __forceinline__ unsigned warp_append(bool want, unsigned* counter) {
    unsigned mask = __ballot_sync(FULL, want);
    unsigned base = 0;
    int leader = __ffs(mask) - 1;
    if (mask && lane_id() == leader) base = atomicAdd(counter, (unsigned)__popc(mask));
    base = __shfl_sync(FULL, base, leader < 0 ? 0 : leader);
    return base + __popc(mask & lanemask_lt());
}

// First index in [lo, hi) of sorted a[] whose value is >= x.
template <typename P>
__device__ __forceinline__ int lower_bound(P a, int lo, int hi, int x) {
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (a[mid] < x)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

// Ranks in (degree, id) order by one block of BINS threads: a stable counting sort on the
// degree, cut at BINS - 1.  Warp w takes a contiguous piece of the n <= 65535 ids, so a bin's
// ids are in order by (warp, round, lane).  The last bin's vertices are then ranked among each
// other directly; false if they are more than TAIL.  hist: BINS / 32 rows of BINS counts in
// shared memory; emit(id, rank, degree) is called once for every id.
template <int BINS, int TAIL, class Emit>
__device__ __forceinline__ bool block_degree_ranks(int n, const uint32_t* deg, uint16_t* hist, Emit emit) {
    static_assert(BINS <= 1024 && TAIL <= BINS, "one bin, or one vertex of the last bin, per thread");
    constexpr int WARPS = BINS / 32;
    __shared__ uint32_t tdeg[TAIL];
    __shared__ int32_t tid_of[TAIL];
    __shared__ int warp_tot[WARPS];
    __shared__ int tail0;
    const int lane = lane_id(), w = threadIdx.x >> 5;
    uint16_t* const mine = hist + w * BINS;  // counts, then the next rank of each bin
    for (int b = lane; b < BINS; b += 32) mine[b] = 0;
    __syncwarp();
    const int chunk = ((n + WARPS - 1) / WARPS + 31) & ~31;
    const int i0 = min(w * chunk, n), i1 = min(i0 + chunk, n);
    for (int b = i0; b < i1; b += 32) {
        const int id = b + lane;
        const int key = id < i1 ? (int)min(deg[id], (uint32_t)BINS - 1) : BINS + lane;
        const unsigned peers = __match_any_sync(FULL, key);
        if (id < i1 && lane == __ffs(peers) - 1) mine[key] = (uint16_t)(mine[key] + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
    int cnt = 0;  // thread b: the bin's vertices, then its first rank
    for (int k = 0; k < WARPS; ++k) cnt += hist[k * BINS + threadIdx.x];
    const int inc = warp_inclusive_scan(cnt);
    if (lane == 31) warp_tot[w] = inc;
    __syncthreads();
    if (w == 0) {
        const int v = lane < WARPS ? warp_tot[lane] : 0;
        const int vi = warp_inclusive_scan(v);
        if (lane < WARPS) warp_tot[lane] = vi - v;
    }
    __syncthreads();
    int base = warp_tot[w] + inc - cnt;
    if (threadIdx.x == BINS - 1) tail0 = base;
    for (int k = 0; k < WARPS; ++k) {
        const int c = hist[k * BINS + threadIdx.x];
        hist[k * BINS + threadIdx.x] = (uint16_t)base;
        base += c;
    }
    __syncthreads();
    const int t0 = tail0;
    for (int b = i0; b < i1; b += 32) {
        const int id = b + lane;
        const uint32_t d = id < i1 ? deg[id] : 0u;
        const int key = id < i1 ? (int)min(d, (uint32_t)BINS - 1) : BINS + lane;
        const unsigned peers = __match_any_sync(FULL, key);
        const int at = id < i1 ? mine[key] : 0;
        __syncwarp();
        if (id < i1) {
            const int r = at + __popc(peers & lanemask_lt());
            if (key < BINS - 1) {
                emit(id, r, d);
            } else if (r - t0 < TAIL) {
                tdeg[r - t0] = d;
                tid_of[r - t0] = id;
            }
            if (lane == __ffs(peers) - 1) mine[key] = (uint16_t)(at + __popc(peers));
        }
        __syncwarp();
    }
    __syncthreads();
    const int k = min(n - t0, TAIL);
    if ((int)threadIdx.x < k) {
        const uint32_t d = tdeg[threadIdx.x];
        int r = t0;
        for (int j = 0; j < k; ++j) r += tdeg[j] < d || (tdeg[j] == d && j < (int)threadIdx.x);
        emit(tid_of[threadIdx.x], r, d);
    }
    __syncthreads();
    return n - t0 <= TAIL;
}

__host__ __device__ __forceinline__ int next_pow2_int(int x) {
    int p = 1;
    while (p < x) p <<= 1;
    return p;
}

}  // namespace tcg

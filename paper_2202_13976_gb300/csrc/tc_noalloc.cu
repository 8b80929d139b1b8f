// tc_count_noalloc: the whole count for a small graph, with every intermediate array in
// a fixed device array of this file, so that the call allocates no memory at all.
//
// Who needs it: code that must not allocate device memory while it runs, for
// example a caller that has handed all free HBM to its own caching allocator, or
// real-time code that forbids allocation after start-up.  The call reads its status
// words back to the host and synchronises the caller's stream before it returns.
//
// The scratch array below is reserved on every GPU that loads the library for as
// long as the process lives (TC_NOALLOC_SCRATCH_BYTES); with lazy module loading the
// runtime places it during the first call on each device, which also loads every kernel
// of this file, so that call belongs at start-up, before the free memory is handed to
// another allocator.  All calls share it and it keeps the previous call's contents;
// the call clears what it needs before use.
// Calls whose work overlaps on the GPU (two streams, or two host threads) race on
// it and give wrong results: the caller must order them.
//
// Seven short kernels, each over as many blocks as its work fills (one for the smallest
// graphs).  One block that did all of it, sorting the pairs as 64-bit keys in global
// memory, took 1.00 ms a call for 30,011 pairs; now 88 us, 46 us of them on the GPU and
// most of these the launches' own 3 us each (262,144 pairs: 220 us).
#include <cuda_runtime.h>

#include <climits>
#include <cstdio>
#include <mutex>

#include "tc_device.cuh"
#include "tc_internal.h"

namespace tcg {
namespace {

constexpr int NA_THREADS = 1024;
constexpr int NA_WARPS = NA_THREADS / 32;
constexpr int64_t NA_MAX_N = TC_NOALLOC_MAX_N;
constexpr int64_t NA_MAX_M = TC_NOALLOC_MAX_M;

// Size of the scratch array in 8-byte words: 16 control words, then per vertex t (8
// bytes) and seven 32-bit arrays, per pair an oriented pair (8 bytes) and an entry.
constexpr int64_t NA_WORDS = 16 + NA_MAX_N + 4 * NA_MAX_N / 2 + NA_MAX_M + (NA_MAX_M + 3 * NA_MAX_N + 2 + 1) / 2;
static_assert(NA_WORDS * 8 == TC_NOALLOC_SCRATCH_BYTES, "scratch size stated in include/tc.h");

static __device__ __align__(256) unsigned long long g_noalloc_scratch[NA_WORDS];

// The arrays of one call, packed for its n and m; the first ones, up to the pairs, start
// at zero.
struct NaArrays {
    unsigned long long* ctl;    // [0] error flags, [3] sum of t
    unsigned long long* t;      // n, by rank
    uint32_t *dmulti, *rowcnt;  // n: non-loop pairs at a vertex (id); pairs of a row (rank)
    uint32_t* dupin;            // n: repeats dropped at a target (rank)
    unsigned long long* pairs;  // m: source | target << 14 | slot in the row << 28, ~0: a loop; then the slots' rows
    int32_t* rowof;             // m: row of every slot of col, -1: freed by a repeat (shares the pairs' memory)
    int32_t* col;               // m
    int32_t* rowstart;          // n + 1
    int32_t* rowlen;            // n
    int32_t* rank;              // n
    int32_t n, m;
    size_t zero_bytes;
};
constexpr int NA_ID_BITS = 14;
static_assert(NA_MAX_N <= 1 << NA_ID_BITS && NA_MAX_M < 1ll << (64 - 2 * NA_ID_BITS), "packed pair");

NaArrays na_arrays(unsigned long long* S, int32_t n, int32_t m) {
    NaArrays A{};
    A.n = n;
    A.m = m;
    A.ctl = S;
    A.t = S + 16;
    A.dmulti = reinterpret_cast<uint32_t*>(A.t + n);
    A.rowcnt = A.dmulti + n;
    A.dupin = A.rowcnt + n;
    A.zero_bytes = (16 + (size_t)n) * 8 + 12 * (size_t)n;
    A.pairs = A.t + n + 2 * (size_t)n;  // four 32-bit arrays' room, of which three are used
    A.rowof = reinterpret_cast<int32_t*>(A.pairs);
    A.col = reinterpret_cast<int32_t*>(A.pairs + m);
    A.rowstart = A.col + m;
    A.rowlen = A.rowstart + n + 1;
    A.rank = A.rowlen + n;
    return A;
}

// Exclusive scan of one value per thread across the block; *total receives the sum.
__device__ int block_scan_excl(int x, int* warp_tot, int* total) {
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int inc = warp_inclusive_scan(x);
    if (lane == 31) warp_tot[w] = inc;
    __syncthreads();
    if (w == 0) {
        const int v = warp_tot[lane];
        const int vi = warp_inclusive_scan(v);
        warp_tot[lane] = vi - v;
        if (lane == 31) *total = vi;
    }
    __syncthreads();
    const int out = warp_tot[w] + inc - x;
    __syncthreads();
    return out;
}

// Degrees of the multigraph (non-loop pairs), id check.  A block counts in shared memory
// (a hub's many increments then cost one global atomic per block).
__device__ void na_degrees(const NaArrays& A, const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                           uint32_t* na_sh, int blk, int blocks) {
    for (int v = threadIdx.x; v < A.n; v += NA_THREADS) na_sh[v] = 0;
    __syncthreads();
    bool bad = false;
    for (int i = blk * NA_THREADS + threadIdx.x; i < A.m; i += blocks * NA_THREADS) {
        const int32_t u = src[i], v = dst[i];
        if ((uint32_t)u >= (uint32_t)A.n || (uint32_t)v >= (uint32_t)A.n) {
            bad = true;
        } else if (u != v) {
            atomicAdd(&na_sh[u], 1u);
            atomicAdd(&na_sh[v], 1u);
        }
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&A.ctl[0], (unsigned long long)ERR_BAD_ID);
    for (int v = threadIdx.x; v < A.n; v += NA_THREADS)
        if (na_sh[v]) atomicAdd(&A.dmulti[v], na_sh[v]);
}

// Ranks in (degree, id) order by one block; the last bin holds at most 2 m / (NA_BINS - 1)
// vertices.
constexpr int NA_BINS = 1024;
constexpr int NA_TAIL = 2 * (int)NA_MAX_M / (NA_BINS - 1) + 1;
static_assert(NA_BINS == NA_THREADS, "one bin per thread");

__device__ void na_rank(const NaArrays& A, uint16_t* na_hist) {
    block_degree_ranks<NA_BINS, NA_TAIL>(A.n, A.dmulti, na_hist, [&](int id, int r, uint32_t) { A.rank[id] = r; });
}

// Oriented pairs, each with its slot in its row.
__device__ void na_count(const NaArrays& A, const int32_t* __restrict__ src, const int32_t* __restrict__ dst, int blk,
                         int blocks) {
    for (int i = blk * (int)blockDim.x + threadIdx.x; i < A.m; i += blocks * (int)blockDim.x) {
        const int32_t u = src[i], v = dst[i];
        unsigned long long p = ~0ull;
        if (u != v) {
            const int32_t a = A.rank[u], b = A.rank[v];
            const int32_t lo = min(a, b), hi = max(a, b);
            const uint32_t slot = atomicAdd(&A.rowcnt[lo], 1u);
            p = (unsigned long long)lo | (unsigned long long)hi << NA_ID_BITS |
                (unsigned long long)slot << 2 * NA_ID_BITS;
        }
        A.pairs[i] = p;
    }
}

// Row starts (every block scans the at most 16,384 row counts for itself, which costs less
// than a launch), then the entries into their slots.
__device__ void na_fill(const NaArrays& A, int32_t* na_start, int blk, int blocks) {  // n words
    __shared__ int warp_tot[NA_WARPS], total;
    const int per = (A.n + NA_THREADS - 1) / NA_THREADS;
    const int r0 = min((int)threadIdx.x * per, A.n), r1 = min(r0 + per, A.n);
    int sum = 0;
    for (int r = r0; r < r1; ++r) sum += (int)A.rowcnt[r];
    int run = block_scan_excl(sum, warp_tot, &total);
    for (int r = r0; r < r1; ++r) {
        na_start[r] = run;
        if (blk == 0) A.rowstart[r] = run;
        run += (int)A.rowcnt[r];
    }
    if (blk == 0 && threadIdx.x == 0) A.rowstart[A.n] = total;
    __syncthreads();
    constexpr unsigned long long ID = (1ull << NA_ID_BITS) - 1;
    for (int i = blk * NA_THREADS + threadIdx.x; i < A.m; i += blocks * NA_THREADS) {
        const unsigned long long p = A.pairs[i];
        if (p != ~0ull) A.col[na_start[p & ID] + (int)(p >> 2 * NA_ID_BITS)] = (int32_t)(p >> NA_ID_BITS & ID);
    }
}

// Sorted distinct rows, a warp each: rows of at most 32 entries by a network across the
// warp, longer ones through a bitmap of the ranks above the row's (any length, any repeats).
constexpr int NA_ROW_WARPS = 8;

__device__ void na_rows(const NaArrays& A, uint32_t* bits, int bm_words, int blk, int blocks) {
    const int lane = lane_id(), w = threadIdx.x >> 5, warps = blockDim.x >> 5;
    uint32_t* const bm = bits + w * bm_words;
    for (int r = blk * warps + w; r < A.n; r += blocks * warps) {
        const int len = (int)A.rowcnt[r], base = A.rowstart[r];
        int kept = 0;
        if (len <= 32) {
            int32_t x = lane < len ? A.col[base + lane] : INT_MAX;
#pragma unroll
            for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
                for (int j = k >> 1; j > 0; j >>= 1) {
                    const int32_t y = __shfl_xor_sync(FULL, x, j);
                    x = ((lane & j) == 0) == ((lane & k) == 0) ? min(x, y) : max(x, y);
                }
            }
            const int32_t prev = __shfl_up_sync(FULL, x, 1);
            const bool keep = lane < len && (lane == 0 || x != prev);
            const unsigned km = __ballot_sync(FULL, keep);
            if (keep)
                A.col[base + __popc(km & lanemask_lt())] = x;
            else if (lane < len)
                atomicAdd(&A.dupin[x], 1u);
            kept = __popc(km);
        } else {
            const int words = (A.n - 1 - r + 31) >> 5;  // ranks r + 1 .. n - 1
            for (int i = lane; i < words; i += 32) bm[i] = 0;
            __syncwarp();
            for (int p = lane; p < len; p += 32) {
                const int off = A.col[base + p] - r - 1;
                const uint32_t bit = 1u << (off & 31);
                if (atomicOr(&bm[off >> 5], bit) & bit) atomicAdd(&A.dupin[off + r + 1], 1u);
            }
            __syncwarp();
            for (int i0 = 0; i0 < words; i0 += 32) {
                uint32_t rest = i0 + lane < words ? bm[i0 + lane] : 0u;
                const int inc = warp_inclusive_scan(__popc(rest));
                int at = base + kept + inc - __popc(rest);
                while (rest) {
                    A.col[at++] = r + 1 + (i0 + lane) * 32 + __ffs(rest) - 1;
                    rest &= rest - 1;
                }
                kept += __shfl_sync(FULL, inc, 31);
            }
            __syncwarp();  // the bitmap is reused by the next row
        }
        if (lane == 0) A.rowlen[r] = kept;
        for (int p = lane; p < len; p += 32) A.rowof[base + p] = p < kept ? r : -1;
    }
}

// Triangles: eight lanes per oriented edge (u, v) look up the entries of the shorter of
// N+(u) after v and N+(v) in the longer.  t[u] += c, t[v] += c and t[w] += 1 for every
// common neighbour w, summed in shared memory per block (a hub takes most of them).
constexpr int NA_TRI_THREADS = 512;

__device__ void na_triangles(const NaArrays& A, uint32_t* na_t, int blk, int blocks) {  // n words
    const int threads = blockDim.x;
    for (int v = threadIdx.x; v < A.n; v += threads) na_t[v] = 0;
    __syncthreads();
    const int gl = threadIdx.x & 7;
    const unsigned gmask = 0xffu << (lane_id() & 24);
    const int slots = A.rowstart[A.n];
    for (int p = (blk * threads + (int)threadIdx.x) >> 3; p < slots; p += (blocks * threads) >> 3) {
        const int u = A.rowof[p];
        if (u < 0) continue;  // a slot freed by a repeat
        const int v = A.col[p];
        const int32_t* a = A.col + p + 1;
        const int la = A.rowstart[u] + A.rowlen[u] - p - 1;
        const int32_t* b = A.col + A.rowstart[v];
        const int lb = A.rowlen[v];
        const int32_t* S = la <= lb ? a : b;
        const int32_t* L = la <= lb ? b : a;
        const int ls = min(la, lb), ll = max(la, lb);
        uint32_t c = 0;
        int lo = 0;  // a lane's keys ascend
        for (int k = gl; k < ls && lo < ll; k += 8) {
            const int32_t x = S[k];
            lo = lower_bound(L, lo, ll, x);
            if (lo < ll && L[lo] == x) {
                atomicAdd(&na_t[x], 1u);
                ++c;
            }
        }
        c += __shfl_xor_sync(gmask, c, 1);
        c += __shfl_xor_sync(gmask, c, 2);
        c += __shfl_xor_sync(gmask, c, 4);
        if (gl == 0 && c) {
            atomicAdd(&na_t[u], c);
            atomicAdd(&na_t[v], c);
        }
    }
    __syncthreads();
    for (int v = threadIdx.x; v < A.n; v += threads)
        if (na_t[v]) atomicAdd(&A.t[v], (unsigned long long)na_t[v]);
}

// Outputs in the caller's ids; sum of t for T.  The simple degree is the distinct
// out-entries plus the in-entries before deduplication less the repeats dropped there.
__device__ void na_outputs(const NaArrays& A, unsigned long long* __restrict__ t_out, double* __restrict__ lcc_out,
                           int blk, int blocks) {
    unsigned long long sum = 0;
    for (int v = blk * (int)blockDim.x + threadIdx.x; v < A.n; v += blocks * (int)blockDim.x) {
        const int32_t r = A.rank[v];
        const unsigned long long tv = A.t[r];
        sum += tv;
        if (t_out) t_out[v] = tv;
        if (lcc_out) {
            const long long d = A.rowlen[r] + (long long)A.dmulti[v] - A.rowcnt[r] - A.dupin[r];
            lcc_out[v] = d < 2 ? 0.0 : __ddiv_rn((double)(2ull * tv), (double)(d * (d - 1)));
        }
    }
    sum = warp_sum(sum);
    if (lane_id() == 0 && sum) atomicAdd(&A.ctl[3], sum);
}

// The phases as kernels; after a bad id the later ones do nothing.
__global__ void __launch_bounds__(NA_THREADS) k_na_degrees(NaArrays A, const int32_t* src, const int32_t* dst) {
    extern __shared__ __align__(16) unsigned char na_sh[];
    na_degrees(A, src, dst, reinterpret_cast<uint32_t*>(na_sh), blockIdx.x, gridDim.x);
}
__global__ void __launch_bounds__(NA_THREADS) k_na_rank(NaArrays A) {
    extern __shared__ __align__(16) unsigned char na_sh[];
    if (A.ctl[0] == 0) na_rank(A, reinterpret_cast<uint16_t*>(na_sh));
}
__global__ void k_na_count(NaArrays A, const int32_t* src, const int32_t* dst) {
    if (A.ctl[0] == 0) na_count(A, src, dst, blockIdx.x, gridDim.x);
}
__global__ void __launch_bounds__(NA_THREADS) k_na_fill(NaArrays A) {
    extern __shared__ __align__(16) unsigned char na_sh[];
    if (A.ctl[0] == 0) na_fill(A, reinterpret_cast<int32_t*>(na_sh), blockIdx.x, gridDim.x);
}
__global__ void __launch_bounds__(NA_ROW_WARPS * 32) k_na_rows(NaArrays A) {
    __shared__ uint32_t bits[NA_ROW_WARPS * NA_MAX_N / 32];
    if (A.ctl[0] == 0) na_rows(A, bits, NA_MAX_N / 32, blockIdx.x, gridDim.x);
}
__global__ void __launch_bounds__(NA_TRI_THREADS) k_na_triangles(NaArrays A) {
    extern __shared__ __align__(16) unsigned char na_sh[];
    if (A.ctl[0] == 0) na_triangles(A, reinterpret_cast<uint32_t*>(na_sh), blockIdx.x, gridDim.x);
}
__global__ void k_na_outputs(NaArrays A, unsigned long long* t_out, double* lcc_out) {
    if (A.ctl[0] == 0) na_outputs(A, t_out, lcc_out, blockIdx.x, gridDim.x);
}

// All phases in one block, for graphs so small that seven launches cost more: the call
// takes 47 us here and 64 us with seven launches for 400 pairs, 64 us both ways for 400
// vertices and 1,600 pairs, 78 and 69 us for 3,000 pairs.
constexpr int NA_ONE_N = 512;
constexpr int NA_ONE_M = 1600;
constexpr int NA_HIST_BYTES = NA_WARPS * NA_BINS * (int)sizeof(uint16_t);
static_assert(NA_WARPS * (NA_ONE_N / 32) * 4 <= NA_HIST_BYTES && NA_ONE_N * 4 <= NA_HIST_BYTES, "shared memory of the phases");

__global__ void __launch_bounds__(NA_THREADS) k_na_one(NaArrays A, const int32_t* src, const int32_t* dst,
                                                       unsigned long long* t_out, double* lcc_out) {
    extern __shared__ __align__(16) unsigned char na_sh[];
    uint32_t* const words = reinterpret_cast<uint32_t*>(na_sh);
    for (int i = threadIdx.x; i < (int)(A.zero_bytes / 4); i += NA_THREADS) reinterpret_cast<uint32_t*>(A.ctl)[i] = 0;
    __syncthreads();
    na_degrees(A, src, dst, words, 0, 1);
    __syncthreads();
    if (A.ctl[0] != 0) return;
    na_rank(A, reinterpret_cast<uint16_t*>(na_sh));
    __syncthreads();
    na_count(A, src, dst, 0, 1);
    __syncthreads();
    na_fill(A, reinterpret_cast<int32_t*>(na_sh), 0, 1);
    __syncthreads();
    na_rows(A, words, NA_ONE_N / 32, 0, 1);
    __syncthreads();
    na_triangles(A, words, 0, 1);
    __syncthreads();
    na_outputs(A, t_out, lcc_out, 0, 1);
}

std::mutex g_na_mutex;
unsigned long long* g_na_ptr[64] = {};

// Once per device: the dynamic shared memory of the kernels (one word per vertex, the
// rank kernel's histograms), which also loads each kernel's code.
cudaError_t na_init() {
    const int word = (int)NA_MAX_N * 4;
    cudaError_t e;
    cudaFuncAttributes a;
    if ((e = cudaFuncSetAttribute(k_na_degrees, cudaFuncAttributeMaxDynamicSharedMemorySize, word)) ||
        (e = cudaFuncSetAttribute(k_na_rank, cudaFuncAttributeMaxDynamicSharedMemorySize, NA_HIST_BYTES)) ||
        (e = cudaFuncSetAttribute(k_na_one, cudaFuncAttributeMaxDynamicSharedMemorySize, NA_HIST_BYTES)) ||
        (e = cudaFuncSetAttribute(k_na_fill, cudaFuncAttributeMaxDynamicSharedMemorySize, word)) ||
        (e = cudaFuncSetAttribute(k_na_triangles, cudaFuncAttributeMaxDynamicSharedMemorySize, word)) ||
        (e = cudaFuncGetAttributes(&a, k_na_count)) || (e = cudaFuncGetAttributes(&a, k_na_rows)))
        return e;
    return cudaFuncGetAttributes(&a, k_na_outputs);
}

}  // namespace
}  // namespace tcg

using namespace tcg;

extern "C" tc_status tc_count_noalloc(int32_t n, int64_t m, const int32_t* src, const int32_t* dst,
                                      uint64_t* T_out, uint64_t* t_out, double* lcc_out, void* cuda_stream) {
    if (!T_out || n < 0 || m < 0 || (m > 0 && (!src || !dst))) return TC_EINVAL;
    if (n > NA_MAX_N || m > NA_MAX_M) return TC_EINVAL;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 64) return TC_ECUDA;
    unsigned long long* S = nullptr;
    {
        // Once per device, with that device current: the device address of the
        // scratch array (its name in host code is not a device address).
        std::lock_guard<std::mutex> lock(g_na_mutex);
        if (!g_na_ptr[dev]) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e == cudaSuccess) e = na_init();
            if (e != cudaSuccess) return TC_ECUDA;
            g_na_ptr[dev] = static_cast<unsigned long long*>(p);
        }
        S = g_na_ptr[dev];
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    if (m == 0) {  // no edge: all counts and coefficients are zero
        if (t_out && n > 0) e = cudaMemsetAsync(t_out, 0, sizeof(uint64_t) * (size_t)n, stream);
        if (e == cudaSuccess && lcc_out && n > 0) e = cudaMemsetAsync(lcc_out, 0, sizeof(double) * (size_t)n, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) return TC_ECUDA;
        *T_out = 0;
        return TC_OK;
    }
    const NaArrays A = na_arrays(S, n, (int32_t)m);
    const size_t word = sizeof(uint32_t) * (size_t)n;
    const auto blocks = [](int64_t work, int64_t per, int64_t most) {
        const int64_t b = (work + per - 1) / per;
        return (unsigned)(b < 1 ? 1 : b > most ? most : b);
    };
    unsigned long long* const t = reinterpret_cast<unsigned long long*>(t_out);
    if (n <= NA_ONE_N && m <= NA_ONE_M) {
        k_na_one<<<1, NA_THREADS, NA_HIST_BYTES, stream>>>(A, src, dst, t, lcc_out);
        count_launch();
    } else {
        e = cudaMemsetAsync(A.ctl, 0, A.zero_bytes, stream);
        if (e != cudaSuccess) return TC_ECUDA;
        // a block of the kernels with a word per vertex takes at least as many pairs as it
        // has words to clear and to flush
        const int64_t share = n > 4096 ? n : 4096;
        k_na_degrees<<<blocks(m, share, 64), NA_THREADS, word, stream>>>(A, src, dst);
        k_na_rank<<<1, NA_THREADS, NA_HIST_BYTES, stream>>>(A);
        k_na_count<<<blocks(m, 256, INT_MAX), 256, 0, stream>>>(A, src, dst);
        k_na_fill<<<blocks(m, share, 64), NA_THREADS, word, stream>>>(A);
        k_na_rows<<<blocks(n, NA_ROW_WARPS, INT_MAX), NA_ROW_WARPS * 32, 0, stream>>>(A);
        k_na_triangles<<<blocks(m, 256, 256), NA_TRI_THREADS, word, stream>>>(A);
        k_na_outputs<<<blocks(n, 256, INT_MAX), 256, 0, stream>>>(A, t, lcc_out);
        count_launch(7);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return TC_ECUDA;
    unsigned long long ctl[4] = {0, 0, 0, 0};
    e = cudaMemcpyAsync(ctl, A.ctl, sizeof(ctl), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return TC_ECUDA;
    if (ctl[0] & ERR_BAD_ID) return TC_EINVAL;
    if (ctl[3] % 3 != 0) return TC_EINTERNAL;
    *T_out = ctl[3] / 3;
    return TC_OK;
}

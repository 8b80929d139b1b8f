// Per-edge set intersection over the degree-oriented CSR (Sec. II-C, Sec. IV-C),
// the planner that splits the edges into buckets, and the final reduction to T
// (Sec. II-C) and LCC (Eq. 2).
//
// Counting rule.  Vertices are ranked by (degree, id) and every oriented row N+(u)
// is sorted and holds only ranks above u.  For the oriented edge (u, v) with
// v = N+(u)[j], the common neighbours are W = N+(u)[j+1 ..] ∩ N+(v): every element
// of N+(v) exceeds v, so only the suffix of N+(u) after v can match.  With c = |W|,
// a triangle {u, v, w} (u < v < w in rank order) is met exactly once, and t[u] += c,
// t[v] += c, t[w] += 1 for every w in W.
//
// Buckets (each oriented edge belongs to exactly one):
//  hub    edges into the highest-ranked vertices ("hubs").  A thread block or a warp
//         stages N+(v) once in shared memory (marks in a table or a bitmap over a window
//         of ranks), then streams the suffix N+(u)[j+1 ..] of every in-edge (u, v)
//         against it, as 16-bit offsets in the window.  This is the on-chip
//         analogue of the paper's caching of remote adjacency lists ranked by degree
//         (Sec. IV-B, Observations 1 and 2): the list that most edges need is read
//         from memory once and reused by all of them.  t[w] increments of the highest
//         ranks are summed in shared memory.
//  small  other edges whose source has 2 <= |N+(u)| <= 256.  HASH (the default): N+(u)
//         becomes a hash set in shared memory, which the rows N+(v) of its edges, laid end
//         to end, are probed in.  Else a group of 8, 16 or 32 lanes stages N+(u) and lane j
//         intersects edge j sequentially, by SSI (Alg. 2) or binary search (Alg. 1), or
//         chosen per edge by Eq. 3.
//  block  other edges whose source has |N+(u)| > 256: one thread block stages N+(u),
//         one warp per edge, methods:
//           MERGE   merge path: the merge of A (suffix) and B = N+(v) is cut into 32
//                   equal diagonal ranges, one per lane, each running Alg. 2
//           SEARCH  every key of A is looked up in B by binary search (Alg. 1)
//           PROBE   every element of B is looked up in A (shared memory) by binary
//                   search; the scan of B stops above max N+(u)
//           BITMAP  like PROBE against a bitmap of N+(u) over its rank window
//           AUTO    Eq. 3 per edge: merge if |B|/|A| <= f (log2|B| - 1) (|A| <= |B|),
//                   else the keys of the shorter list are searched in the longer
#include <climits>
#include <type_traits>

#include "tc_device.cuh"
#include "tc_internal.h"

namespace tcg {

namespace {

constexpr int THREADS = 256;
constexpr int SMALL_WARPS = 8;         // warps per block in the small-bucket kernel
constexpr int SMALL_BLOCKS = 8;        // its resident blocks per SM (the grid is one wave of them)
constexpr int SMALL_WIDE_MAX = 256;    // longest N+(u) the warp-per-source kernel stages
constexpr int HASH_LG_SHORT = 8;       // slots of the hash kernel's sets (log2): sources of at most 32 entries,
constexpr int HASH_LG_WIDE = 9;        // and of at most SMALL_WIDE_MAX
constexpr int HASH_CUT = 64;           // rows longer than this are cut at max N+(u) by the hash kernel
constexpr int CTA_THREADS = 256;       // block push kernel
constexpr int CTA_WARPS = CTA_THREADS / 32;
constexpr int CTA_LIST_MAX = 2048;     // staged list capacity of the block push kernel
constexpr int BITMAP_WORDS = 4096;     // its bitmap window: 131072 ranks
constexpr int HUB_THREADS = 256;
constexpr int HUB_WARPS = HUB_THREADS / 32;
constexpr int HUB_BM_WORDS = HUB_BM_BITS / 32;
constexpr int HUB_CNT_MAX = 1024;      // hub lists longer than this count matches globally
constexpr int HUB_BLOCKS = 6;          // resident blocks of the hub kernel per SM (registers and shared memory)
constexpr int HUB_WARP_MAX = 256;      // longest N+(v) a single warp stages
constexpr int HUB_HASH_LOAD = 2;       // its hash table has at least this many slots per key
constexpr int HUB_HASH_MAX = HUB_HASH_LOAD * HUB_WARP_MAX;
constexpr int SCAT_STEPS = 4;          // lockstep steps of the row-walk scatter in flight together
constexpr int HUB_BATCH = 32;          // in-edges per batch of a big hub
constexpr int HUB_LONG = 16;           // suffixes at least this long are read by lane groups
constexpr int HUB_GROUPS = 4;          // long suffixes one warp reads at a time
constexpr int HUB_GLANES = 32 / HUB_GROUPS;
constexpr int HUB_UNROLL = 8;          // entries a lane reads per round of a long suffix

struct Sink {
    uint32_t* cnt;               // per-position counters (shared), or null
    unsigned long long* t;       // global counts, used when cnt is null
    const int32_t* Lu;           // N+(u) (shared or global)
    uint32_t* supA;              // per-edge support of the entries of N+(u) when cnt is null, or null
    uint32_t* supB;              // per-edge support of the entries of N+(v), or null
    __device__ __forceinline__ void hit(int p) const {
        if (cnt) {
            atomicAdd(&cnt[p], 1u);
        } else {
            atomicAdd(&t[Lu[p]], 1ull);
            if (supA) atomicAdd(&supA[p], 1u);
        }
    }
    __device__ __forceinline__ void hitB(int k) const {
        if (supB) atomicAdd(&supB[k], 1u);
    }
};

// Number of elements of sorted B[0, b) that are <= x.
__device__ __forceinline__ int count_le(const int32_t* __restrict__ B, int b, int32_t x) {
    int lo = 0, hi = b;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (B[mid] <= x)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

__device__ __forceinline__ bool eq3_prefers_merge(int a, int b, float factor) {
    int s = min(a, b), l = max(a, b);
    return (float)l <= factor * (log2f((float)l) - 1.0f) * (float)s;
}

// Lane-per-edge choice between the batched merge and binary search: Eq. 3, except
// that an N+(v) of at most 16 entries (two 8-entry loads of the merge) is always
// merged, since one merge round costs less than the dependent loads of a search.
__device__ __forceinline__ int small_auto(int a, int dv, float factor) {
    return dv <= 16 || eq3_prefers_merge(a, dv, factor) || dv < a ? TC_STRAT_MERGE : TC_STRAT_SEARCH;
}

// ---- warp-cooperative methods (block push kernel) -----------------------------

__device__ uint32_t edge_merge(const Sink& S, int a0, int du, const int32_t* __restrict__ B, int b) {
    const int lane = lane_id();
    const int32_t* A = S.Lu + a0;
    const int a = du - a0;
    b = count_le(B, b, A[a - 1]);  // elements of B above max(A) cannot match
    const int64_t total = (int64_t)a + b;
    const int d0 = (int)((total * lane) >> 5);
    const int d1 = (int)((total * (lane + 1)) >> 5);
    int lo = max(0, d0 - b), hi = min(d0, a);
    while (lo < hi) {  // A elements among the first d0 merged items (ties: A first)
        int mid = (lo + hi) >> 1;
        if (A[mid] <= B[d0 - mid - 1])
            lo = mid + 1;
        else
            hi = mid;
    }
    int i = lo, j = d0 - lo;
    int32_t bj = j < b ? B[j] : INT_MAX;
    uint32_t c = 0;
    for (int step = d0; step < d1; ++step) {
        if (i < a && A[i] <= bj) {
            if (A[i] == bj) {
                S.hit(a0 + i);
                S.hitB(j);
                ++c;
            }
            ++i;
        } else {
            ++j;
            bj = j < b ? B[j] : INT_MAX;
        }
    }
    return warp_sum(c);
}

__device__ uint32_t edge_search(const Sink& S, int a0, int du, const int32_t* __restrict__ B, int b) {
    const int lane = lane_id();
    uint32_t c = 0;
    int lo = 0;
    for (int k = a0 + lane; k < du; k += 32) {
        int32_t y = S.Lu[k];
        int p = lower_bound(B, lo, b, y);
        lo = p;  // keys of this lane increase
        if (p < b && B[p] == y) {
            S.hit(k);
            S.hitB(p);
            ++c;
        }
    }
    return warp_sum(c);
}

__device__ uint32_t edge_probe(const Sink& S, int a0, int du, const int32_t* __restrict__ B, int b) {
    const int lane = lane_id();
    const int32_t maxu = S.Lu[du - 1];
    uint32_t c = 0;
    for (int k0 = 0; k0 < b; k0 += 32) {
        int k = k0 + lane;
        int32_t x = k < b ? B[k] : INT_MAX;
        if (x <= maxu) {
            int p = lower_bound(S.Lu, a0, du, x);
            if (S.Lu[p] == x) {  // p < du because x <= max
                S.hit(p);
                S.hitB(k);
                ++c;
            }
        }
        if (__any_sync(FULL, x > maxu)) break;  // B is sorted: later chunks exceed too
    }
    return warp_sum(c);
}

// Bitmap over ranks (u, maxu]: bit (x - u - 1) set iff x in N+(u); pre[w] = number of
// set bits in the words before w, i.e. the position in N+(u) of the word's first member.
__device__ uint32_t edge_bitmap(const uint32_t* bm, const uint16_t* pre, int32_t u, int32_t maxu,
                                uint32_t* cnt, const int32_t* __restrict__ B, int b, uint32_t* __restrict__ supB) {
    const int lane = lane_id();
    uint32_t c = 0;
    for (int k0 = 0; k0 < b; k0 += 32) {
        int k = k0 + lane;
        int32_t x = k < b ? B[k] : INT_MAX;
        if (x <= maxu) {
            int off = x - u - 1;
            uint32_t w = bm[off >> 5], bit = 1u << (off & 31);
            if (w & bit) {
                atomicAdd(&cnt[pre[off >> 5] + __popc(w & (bit - 1))], 1u);
                if (supB) atomicAdd(&supB[k], 1u);
                ++c;
            }
        }
        if (__any_sync(FULL, x > maxu)) break;
    }
    return warp_sum(c);
}

__device__ __forceinline__ uint32_t edge_dispatch(int method, const Sink& S, int a0, int du,
                                                  const int32_t* __restrict__ B, int b) {
    switch (method) {
        case TC_STRAT_MERGE: return edge_merge(S, a0, du, B, b);
        case TC_STRAT_SEARCH: return edge_search(S, a0, du, B, b);
        default: return edge_probe(S, a0, du, B, b);
    }
}

// Builds the bitmap of the staged list L[0, d) over ranks (base, base + 32 W] and its
// per-word prefix counts; a whole block calls it.
template <int THREADS_>
__device__ void build_bitmap(uint32_t* bm, uint16_t* pre, uint32_t* slice, const int32_t* __restrict__ L, int d,
                             int32_t base, int W) {
    const int lane = lane_id(), w = threadIdx.x >> 5;
    constexpr int WARPS = THREADS_ / 32;
    for (int i = threadIdx.x; i < W; i += THREADS_) bm[i] = 0;
    __syncthreads();
    for (int p = threadIdx.x; p < d; p += THREADS_) {
        int off = L[p] - base - 1;
        atomicOr(&bm[off >> 5], 1u << (off & 31));
    }
    __syncthreads();
    // exclusive prefix of per-word popcounts: within 32-word slices (one warp each),
    // then over slice totals (warp 0), then the slice offsets are added
    const int slices = (W + 31) >> 5;
    for (int s = w; s < slices; s += WARPS) {
        const int i = s * 32 + lane;
        const int pc = i < W ? __popc(bm[i]) : 0;
        const int inc = warp_inclusive_scan(pc);
        if (i < W) pre[i] = (uint16_t)(inc - pc);
        if (lane == 31) slice[s] = (uint32_t)inc;
    }
    __syncthreads();
    if (w == 0) {
        uint32_t carry = 0;
        for (int c0 = 0; c0 < slices; c0 += 32) {
            const int i = c0 + lane;
            const uint32_t v = i < slices ? slice[i] : 0u;
            const uint32_t inc = warp_inclusive_scan(v);
            if (i < slices) slice[i] = carry + inc - v;
            carry += __shfl_sync(FULL, inc, 31);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < W; i += THREADS_) pre[i] = (uint16_t)(pre[i] + slice[i >> 5]);
    __syncthreads();
}

// ---- lane-sequential methods (small bucket) -----------------------------------
// A = Lu[a0, du) (shared, sorted), B = N+(v) (global, sorted).  A match at position
// p of Lu adds one to cnt[p].

// Merge with B read eight entries at a time (independent loads), A in shared memory.
__device__ uint32_t lane_merge_batched(const int32_t* Lu, int a0, int du, const int32_t* __restrict__ B, int b,
                                       uint32_t* cnt) {
    uint32_t c = 0;
    int i = a0;
    const int32_t mx = Lu[du - 1];
    for (int k0 = 0; k0 < b && i < du; k0 += 8) {
        int32_t y[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) y[q] = k0 + q < b ? B[k0 + q] : INT_MAX;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            while (i < du && Lu[i] < y[q]) ++i;
            if (i < du && Lu[i] == y[q]) {
                atomicAdd(&cnt[i], 1u);
                ++c;
                ++i;
            }
        }
        if (y[7] >= mx) break;
    }
    return c;
}

// keys of A looked up in B
__device__ uint32_t lane_search(const int32_t* Lu, int a0, int du, const int32_t* __restrict__ B, int b,
                                uint32_t* cnt) {
    uint32_t c = 0;
    int lo = 0;
    for (int i = a0; i < du && lo < b; ++i) {
        const int32_t x = Lu[i];
        const int p = lower_bound(B, lo, b, x);
        lo = p;
        if (p < b && B[p] == x) {
            atomicAdd(&cnt[i], 1u);
            ++c;
        }
    }
    return c;
}

// keys of B looked up in A
__device__ uint32_t lane_search_rev(const int32_t* Lu, int a0, int du, const int32_t* __restrict__ B, int b,
                                    uint32_t* cnt) {
    uint32_t c = 0;
    int lo = a0;
    const int32_t mx = Lu[du - 1];
    for (int k = 0; k < b && lo < du; ++k) {
        const int32_t y = B[k];
        if (y > mx) break;
        const int p = lower_bound(Lu, lo, du, y);
        lo = p;
        if (p < du && Lu[p] == y) {
            atomicAdd(&cnt[p], 1u);
            ++c;
        }
    }
    return c;
}

// ---- planner -----------------------------------------------------------------

// Hub candidates; the block that counts last sets the hub count and the core's size.
__global__ void k_hub_count(int32_t n, const int32_t* __restrict__ deg, int min_degree, int32_t hub_cap, int hub_max,
                            int core_max, DevStats* stats) {
    __shared__ unsigned sum;
    if (threadIdx.x == 0) sum = 0;
    __syncthreads();
    unsigned c = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += stride)
        c += deg[r] >= min_degree ? 1u : 0u;
    c = __reduce_add_sync(FULL, c);
    if (lane_id() == 0 && c) atomicAdd(&sum, c);
    __syncthreads();
    if (threadIdx.x != 0) return;
    if (sum) atomicAdd(&stats->hub_candidates, sum);
    __threadfence();
    if (atomicAdd(&stats->hub_blocks, 1u) == gridDim.x - 1) {
        unsigned k = atomicAdd(&stats->hub_candidates, 0u);
        k = min(k, (unsigned)hub_max);
        k = min(k, (unsigned)hub_cap);
        stats->hub_count = k;
        stats->core_n = min(k, (unsigned)core_max);
    }
}

// In-degree d-(v) = deg(v) - d+(v) of every hub slot (0 for slots below the hubs),
// less the in-edges from the dense core, which the core count covers.
__global__ void k_hub_indeg(int32_t n, int32_t hub_cap, const int32_t* __restrict__ deg,
                            const int32_t* __restrict__ rowlen, const uint32_t* __restrict__ core_cnt,
                            uint32_t* __restrict__ cnt, DevStats* stats) {
    const int32_t R = n - (int32_t)stats->hub_count;
    const int32_t c0 = n - (int32_t)stats->core_n;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < hub_cap; i += stride) {
        const int32_t r = n - hub_cap + (int32_t)i;
        uint32_t d = r >= R ? (uint32_t)(deg[r] - rowlen[r]) : 0u;
        if (r >= c0) d -= core_cnt[r - c0];
        cnt[i] = d;
    }
}

// The hub in-edge records are written by tiles of entries (k_row_of, k_hub_scatter)
// when the hub in-edges are at least a quarter of the entries of the non-core rows,
// else by a walk over the rows' hub tails (k_hub_scatter_rows).  All three kernels
// are launched and read the choice from the planned counts.
__device__ __forceinline__ bool scatter_by_tiles(const int64_t* __restrict__ hub_start, int32_t hub_cap,
                                                 const int64_t* __restrict__ rowstart, int32_t c0) {
    return 4 * hub_start[hub_cap] >= rowstart[c0];
}

// Source row of every entry of the counted non-core rows (whole row capacity, so that the
// slots left free by deduplication also name a valid row).  A lane writes its own
// row when it holds at most 32 entries; longer rows are written by the whole warp.
__global__ void k_row_of(int32_t n, int32_t hub_cap, const int64_t* __restrict__ rowstart,
                         const int64_t* __restrict__ hub_start, int32_t* __restrict__ rowof, int32_t src_lo,
                         int32_t src_hi, const DevStats* stats) {
    const int32_t c0 = n - (int32_t)stats->core_n;
    if (!scatter_by_tiles(hub_start, hub_cap, rowstart, c0)) return;
    const int lane = lane_id();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int32_t end = min(src_hi, c0);
    // the loop bound is uniform across a warp, as the ballot needs all 32 lanes
    for (int64_t b = src_lo + (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); b < end; b += stride) {
        const int64_t u = b + lane;
        const int64_t a0 = u < end ? rowstart[u] : 0, a1 = u < end ? rowstart[u + 1] : 0;
        const bool longrow = a1 - a0 > 32;
        if (!longrow)
            for (int64_t p = a0; p < a1; ++p) rowof[p] = (int32_t)u;
        unsigned lm = __ballot_sync(FULL, longrow);
        while (lm) {
            const int r = __ffs(lm) - 1;
            lm &= lm - 1;
            const int64_t ar = __shfl_sync(FULL, a0, r), br = __shfl_sync(FULL, a1, r);
            for (int64_t p = ar + lane; p < br; p += 32) rowof[p] = (int32_t)(b + r);
        }
    }
}

// Window entries.  The ranks are read in windows from the top: HUB_WIN ranks in window
// 1, where most suffix entries lie (R-MAT scale 20 / 23: 98% / 91% of what the hub bucket
// probes), then two windows of HUB_WIN2, which reach below every hub.  Each non-core
// row's entries from the lowest hub on are kept once more as 16-bit offsets in their
// window, eight to a 16-byte vector; a row's windows start a vector each, from the
// first on, and are padded with the offset that no hub marks.  A block takes 256
// consecutive rows, reserves their vectors with one atomic and writes them a thread
// per vector.
constexpr int WIN_THREADS = 256;
constexpr int WINS = 3;

struct Windows {
    int32_t first[WINS + 1];  // first rank of window k
    explicit Windows(int32_t n) {
        first[0] = n;
        first[1] = n < HUB_WIN ? 0 : n - HUB_WIN;
        for (int k = 2; k <= WINS; ++k) first[k] = first[k - 1] < HUB_WIN2 ? 0 : first[k - 1] - HUB_WIN2;
    }
};
static_assert(HUB_WIN + (WINS - 1) * HUB_WIN2 >= HUB_BM_BITS, "the windows reach below every hub");

__device__ __forceinline__ uint32_t vectors_of(uint32_t entries) { return (entries + 7u) >> 3; }

// The place of window 1's rank i among its counters.  Neighbouring ranks' suffixes hold runs
// of consecutive ranks in graphs whose ids have locality; the lanes of a probe are then
// eight ranks apart, in four banks if the places were the ranks themselves.  Its own inverse.
__host__ __device__ __forceinline__ constexpr uint32_t win_place(uint32_t i) { return i ^ ((i >> 5) & 7u); }
constexpr uint32_t WIN_NONE = 4 * win_place(HUB_WIN);  // the offset that no hub marks
constexpr bool win_places_ok() {
    for (uint32_t i = 0; i <= HUB_WIN; ++i)
        if (win_place(i) > HUB_WIN || win_place(win_place(i)) != i || win_place(i) >> 3 != i >> 3) return false;
    return true;
}
static_assert((HUB_WIN & 7) == 7 && win_places_ok(), "a permutation of each group of eight");

// A row's place in the windows below the first: {first vector of window 2, entries in
// window 1, entries in window 2 | in window 3 << 16, 0}.
__device__ __forceinline__ uint32_t low_len(const uint4& r, int k) { return k == 2 ? r.z & 0xffffu : r.z >> 16; }

__global__ void __launch_bounds__(WIN_THREADS) k_win_build(int32_t n, Windows T, const int2* __restrict__ rowinfo,
                                                           const int32_t* __restrict__ col,
                                                           uint2* __restrict__ winrow, uint4* __restrict__ winlow,
                                                           uint4* __restrict__ win, int64_t win_cap, int32_t src_lo,
                                                           int32_t src_hi, DevStats* stats) {
    __shared__ uint32_t pref[WIN_THREADS];
    __shared__ int32_t cut[WINS + 1][WIN_THREADS];  // the row's end, then where its windows 1, 2, ... start in col
    __shared__ uint32_t wtot[WIN_THREADS / 32];
    __shared__ uint32_t base_sh;
    const int32_t c0 = n - (int32_t)stats->core_n;
    const int32_t R = n - (int32_t)stats->hub_count;
    const int lane = lane_id(), w = threadIdx.x >> 5;
    if (stats->hub_count == 0) return;
    for (int64_t t0 = (int64_t)blockIdx.x * WIN_THREADS; t0 < c0; t0 += (int64_t)gridDim.x * WIN_THREADS) {
        const int64_t u = t0 + threadIdx.x;
        uint32_t nv = 0, len[WINS + 1] = {};
        // a row without a hub has no in-edge records, one of a single entry no suffix: nothing
        // here is read for them (but for the hubs' own lists)
        bool hubrow = false;
        if (u < c0 && ((u >= src_lo && u < src_hi) || u >= R)) {  // a shard: its sources and the hubs
            const int2 ri = rowinfo[u];
            const int32_t end = ri.x + ri.y;
            hubrow = ri.y > (u < R ? 1 : 0) && col[end - 1] >= R;
            if (hubrow) {
                int at = ri.y;
                cut[0][threadIdx.x] = end;
#pragma unroll
                for (int k = 1; k <= WINS; ++k) {
                    const int hi = at;
                    if (at > 0 && R < T.first[k - 1] && col[ri.x + at - 1] >= R)
                        at = lower_bound(col + ri.x, 0, at, max(T.first[k], R));
                    cut[k][threadIdx.x] = ri.x + at;
                    len[k] = (uint32_t)(hi - at);
                    nv += vectors_of(len[k]);
                }
                // sources outside the shard, and rows of one entry, have no suffix to read
                if (u < src_lo || u >= src_hi || ri.y < 2) nv = 0;
            }
        }
        const uint32_t inc = warp_inclusive_scan(nv);
        if (lane == 31) wtot[w] = inc;
        __syncthreads();
        uint32_t before = 0, total = 0;
#pragma unroll
        for (int k = 0; k < WIN_THREADS / 32; ++k) {
            before += k < w ? wtot[k] : 0;
            total += wtot[k];
        }
        if (threadIdx.x == 0) base_sh = total ? atomicAdd(&stats->win_vecs, total) : 0u;
        pref[threadIdx.x] = before + inc - nv;
        __syncthreads();
        const uint32_t base = base_sh;
        if (hubrow) {
            const uint32_t v0 = base + before + inc - nv;
            winrow[u] = make_uint2(v0, len[1]);
            if (R < T.first[1])
                winlow[u] = make_uint4(v0 + vectors_of(len[1]), len[1], len[2] | len[3] << 16, 0);
        }
        for (uint32_t k = threadIdx.x; k < total; k += WIN_THREADS) {
            int lo = 0;  // the last row whose vectors start at or before k
#pragma unroll
            for (int step = WIN_THREADS / 2; step > 0; step >>= 1)
                if (pref[lo + step] <= k) lo += step;
            uint32_t rel = k - pref[lo];
            int win_no = 1;
            int32_t p1 = cut[0][lo], p0 = cut[1][lo];
            while (win_no < WINS && rel >= vectors_of(p1 - p0)) {
                rel -= vectors_of(p1 - p0);
                p1 = p0;
                p0 = cut[++win_no][lo];
            }
            const int32_t first = win_no == 1 ? T.first[1] : win_no == 2 ? T.first[2] : T.first[3];
            const uint32_t none = win_no == 1 ? WIN_NONE : (uint32_t)HUB_WIN2;
            uint32_t o[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int64_t p = (int64_t)p0 + 8 * (int64_t)rel + j;
                o[j] = none;
                if (p < p1) {
                    const uint32_t i = (uint32_t)(col[p] - first);
                    o[j] = win_no == 1 ? 4u * win_place(i) : i;
                }
            }
            if ((int64_t)base + k < win_cap)  // always true: win_vec_cap
                win[base + k] = make_uint4(o[0] | o[1] << 16, o[2] | o[3] << 16, o[4] | o[5] << 16, o[6] | o[7] << 16);
            else
                atomicOr(&stats->err, ERR_OVERFLOW);
        }
        __syncthreads();  // the shared arrays are reused by the next rows
    }
}

// Every oriented entry (u -> v) of a row outside the dense core with v a hub becomes
// an in-edge record of v: {u, entries of N+(u) after v}, one 8-byte store into v's
// segment (R-MAT scale 23: 0.83 ms; 16-byte records that also named the suffix's place
// took 1.26 ms, so the hub kernels gather that place by u).  Blocks take tiles of
// SCAT_TILE consecutive entries (16 bytes per thread and load), so the work is spread
// evenly whatever the row lengths;
// entries in the slots deduplication left free are skipped.  The SCAT_TOP highest
// hubs, whose cursors every tile would contend for, are served per tile: shared-
// memory counters give each entry its offset, then one global atomic per hub and
// tile reserves the tile's run; the other hubs take their slot from a global
// cursor per entry.  Records of one tile stay together, nearly in source order.
constexpr int SCAT_THREADS = 1024;  // 256 take 4 to 8 % longer (more reservations)
constexpr int SCAT_ITEMS = 8;  // entries per thread and tile (two 16-byte loads)
constexpr int SCAT_TILE = SCAT_THREADS * SCAT_ITEMS;
constexpr int SCAT_TOP = 2048;

__global__ void __launch_bounds__(SCAT_THREADS) k_hub_scatter(int32_t n, int32_t hub_cap,
                                                              const int64_t* __restrict__ rowstart,
                                                              const int2* __restrict__ rowinfo,
                                                              const int32_t* __restrict__ col,
                                                              const int32_t* __restrict__ rowof,
                                                              const int64_t* __restrict__ hub_start,
                                                              unsigned long long* __restrict__ cur,
                                                              uint2* __restrict__ in_rec, int32_t src_lo,
                                                              int32_t src_hi, DevStats* stats) {
    __shared__ uint32_t lcnt[SCAT_TOP];
    __shared__ uint32_t gbase[SCAT_TOP];  // slots are below 2^31
    const int32_t R = n - (int32_t)stats->hub_count;
    const int32_t c0 = n - (int32_t)stats->core_n;  // rows of the dense core are counted there
    const int top = min((int)stats->hub_count, SCAT_TOP);
    const int32_t T0 = n - top;  // top hubs: ranks T0 .. n-1 (all hubs)
    const int32_t H0 = n - hub_cap;  // rank of hub slot 0
    if (!scatter_by_tiles(hub_start, hub_cap, rowstart, c0)) return;
    // the entries of the counted rows
    const int64_t mbeg = rowstart[min(src_lo, c0)], mend = rowstart[min(src_hi, c0)];
    const int64_t total = hub_start[hub_cap];
    for (int64_t t0 = (mbeg & ~(int64_t)3) + (int64_t)blockIdx.x * SCAT_TILE; t0 < mend; t0 += (int64_t)gridDim.x * SCAT_TILE) {
        for (int h = threadIdx.x; h < top; h += SCAT_THREADS) lcnt[h] = 0;
        __syncthreads();
        int32_t x[SCAT_ITEMS], u[SCAT_ITEMS], len[SCAT_ITEMS];
        uint32_t loc[SCAT_ITEMS];
#pragma unroll
        for (int k = 0; k < SCAT_ITEMS / 4; ++k) {
            const int64_t e0 = t0 + ((int64_t)k * SCAT_THREADS + threadIdx.x) * 4;
            if (e0 + 3 < mend) {
                const int4 q = *reinterpret_cast<const int4*>(col + e0);
                x[4 * k] = q.x, x[4 * k + 1] = q.y, x[4 * k + 2] = q.z, x[4 * k + 3] = q.w;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) x[4 * k + j] = e0 + j < mend ? col[e0 + j] : -1;
            }
        }
#pragma unroll
        for (int e = 0; e < SCAT_ITEMS; ++e) {
            const int64_t p = t0 + ((int64_t)(e >> 2) * SCAT_THREADS + threadIdx.x) * 4 + (e & 3);
            if (p < mbeg) x[e] = -1;
            if (x[e] >= R) {
                u[e] = rowof[p];
                const int2 ri = rowinfo[u[e]];
                len[e] = (int32_t)((int64_t)ri.x + ri.y - p - 1);
                if (len[e] < 0) x[e] = -1;  // a slot freed by deduplication
            }
        }
        // the slot reservations of all items first, so that their round trips overlap,
        // then the records of the hubs below the top ones
        uint32_t gslot[SCAT_ITEMS];
#pragma unroll
        for (int e = 0; e < SCAT_ITEMS; ++e) {
            gslot[e] = 0;
            if (x[e] >= T0)
                loc[e] = atomicAdd(&lcnt[x[e] - T0], 1u);
            else if (x[e] >= R)
                gslot[e] = (uint32_t)atomicAdd(&cur[x[e] - H0], 1ull);
        }
#pragma unroll
        for (int e = 0; e < SCAT_ITEMS; ++e) {
            if (x[e] < R || x[e] >= T0) continue;
            if ((int64_t)gslot[e] < total)  // counts and entries disagree only on a bug: never write outside
                in_rec[gslot[e]] = make_uint2((uint32_t)u[e], (uint32_t)len[e]);
            else
                atomicOr(&stats->err, ERR_OVERFLOW);
        }
        __syncthreads();
        for (int h = threadIdx.x; h < top; h += SCAT_THREADS) {
            const uint32_t c = lcnt[h];
            if (c) gbase[h] = (uint32_t)atomicAdd(&cur[T0 + h - H0], (unsigned long long)c);
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < SCAT_ITEMS; ++e) {
            if (x[e] < T0) continue;
            const uint32_t slot = gbase[x[e] - T0] + loc[e];
            if (slot < total)
                in_rec[slot] = make_uint2((uint32_t)u[e], (uint32_t)len[e]);
            else
                atomicOr(&stats->err, ERR_OVERFLOW);
        }
        __syncthreads();  // lcnt and gbase are reused by the next tile
    }
}

// The same records when hub entries are a small share of the entries (flat degree
// distributions): a warp takes 32 consecutive rows (one per lane) and walks their
// hub tails from the end backwards in lockstep, so rows without a hub cost one
// load; the highest-ranked hubs end almost every row, so lanes that name the same
// hub in a step reserve their slots with one atomic.
__global__ void k_hub_scatter_rows(int32_t n, int32_t hub_cap, const int64_t* __restrict__ rowstart,
                                   const int32_t* __restrict__ rowlen, const int32_t* __restrict__ col,
                                   const int64_t* __restrict__ hub_start, unsigned long long* __restrict__ cur,
                                   uint2* __restrict__ in_rec, int32_t src_lo, int32_t src_hi,
                                   DevStats* stats) {
    const int32_t R = n - (int32_t)stats->hub_count;
    const int32_t c0 = n - (int32_t)stats->core_n;  // rows of the dense core are counted there
    if (scatter_by_tiles(hub_start, hub_cap, rowstart, c0)) return;
    const int64_t total = hub_start[hub_cap];
    const int lane = lane_id();
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int32_t end = min(src_hi, c0);  // of the counted rows
    for (int64_t w0 = src_lo + (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; w0 < end;
         w0 += warps * 32) {
        const int64_t u = w0 + lane;
        const int du = u < end ? rowlen[u] : 0;
        const int64_t base = u < n ? rowstart[u] : 0;
        int p = du - 1;
        // SCAT_STEPS steps at a time: their loads, then their slot reservations, are
        // independent and in flight together.  Walking backwards, the hub entries of a
        // row come first, so a lane's active steps are a prefix.
        for (int step = 0;; step += SCAT_STEPS) {
            int32_t x[SCAT_STEPS];
#pragma unroll
            for (int j = 0; j < SCAT_STEPS; ++j) x[j] = p - j >= 0 ? col[base + p - j] : -1;
            if (!__any_sync(FULL, x[0] >= R)) break;
            unsigned peers[SCAT_STEPS];
            int64_t slot0[SCAT_STEPS];
#pragma unroll
            for (int j = 0; j < SCAT_STEPS; ++j) {
                const bool active = x[j] >= R;
                // the first steps meet the most contended (highest) hubs: aggregate them;
                // afterwards every lane reserves its own slot
                peers[j] = __match_any_sync(FULL, active && step + j < 16 ? x[j] : -1 - lane);
                slot0[j] = 0;
                if (active && lane == __ffs(peers[j]) - 1)
                    slot0[j] = (int64_t)atomicAdd(&cur[x[j] - (n - hub_cap)], (unsigned long long)__popc(peers[j]));
            }
#pragma unroll
            for (int j = 0; j < SCAT_STEPS; ++j) {
                slot0[j] = __shfl_sync(FULL, slot0[j], __ffs(peers[j]) - 1);
                if (x[j] >= R) {
                    const int64_t slot = slot0[j] + __popc(peers[j] & lanemask_lt());
                    if (slot < total)  // counts and entries disagree only on a bug: never write outside
                        in_rec[slot] = make_uint2((uint32_t)u, (uint32_t)(du - 1 - (p - j)));
                    else
                        atomicOr(&stats->err, ERR_OVERFLOW);
                }
            }
            p = x[SCAT_STEPS - 1] >= R ? p - SCAT_STEPS : -1;
        }
    }
}

// Work lists of the hubs (hub 0 = highest rank).  A hub is big when its in-degree
// reaches big_in or its list is too long for one warp.  Its in-edges are cut into
// slices: a window task is {v, first in-edge, first entry of N+(v) in window 1,
// in-edges | entries there << TASK_BITS}; a below-window task {v, first in-edge,
// in-edges, entries of N+(v) below window 1}.  One atomic per list and warp keeps the
// lists nearly in rank order (blocks start in order), which is all the work queues need.
constexpr int TASK_BITS = 12;
static_assert(HUB_SLICE < 1 << TASK_BITS && (int64_t)HUB_WIN << TASK_BITS < INT_MAX, "window task fields");

// Per-edge support: the part below window 1 of a big hub's list is taken by a block from so
// many entries on (a long one has to be: HUB_WARP_MAX).  Block + warp kernel, from 0 / 64 /
// 256 entries on: G(60,000) of 16.8 M pairs 1.34 + 0.03, 1.19 + 1.05, 0.37 + 3.58 ms; R-MAT
// scale 20 54 + 127, 3 + 151, 3 + 150 us.
constexpr int HUB_LIST_MIN = 64;
static_assert(HUB_LIST_MIN <= HUB_WARP_MAX, "what a warp stages");

// First of `mine` slots reserved for this lane in a list (a warp's lanes in order).
__device__ __forceinline__ unsigned warp_reserve(unsigned mine, unsigned* counter) {
    const unsigned inc = warp_inclusive_scan(mine);
    const unsigned tot = __shfl_sync(FULL, inc, 31);
    unsigned base = 0;
    if (lane_id() == 0 && tot) base = atomicAdd(counter, tot);
    return __shfl_sync(FULL, base, 0) + inc - mine;
}

__global__ void k_hub_lists(int32_t n, int32_t hub_cap, int32_t T0w, const int2* __restrict__ rowinfo,
                            const int32_t* __restrict__ col, const uint2* __restrict__ winrow,
                            const uint32_t* __restrict__ indeg, const int64_t* __restrict__ hub_start, int big_in,
                            int32_t* __restrict__ big_list, int32_t* __restrict__ long_list,
                            int4* __restrict__ win_task, int4* __restrict__ low_task, int64_t task_cap,
                            const unsigned long long* __restrict__ cur, bool shard, DevStats* stats) {
    const int64_t K = stats->hub_count;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int lane = lane_id();
    // the loop bound is uniform across a warp, as the appends need all 32 lanes
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); b < K; b += stride) {
        const int64_t i = b + lane;
        const int32_t v = n - 1 - (int32_t)i;
        bool big = false;
        uint32_t din = 0;
        int dlow = 0, dwin = 0;
        int2 ri = make_int2(0, 0);
        int64_t e0 = 0;
        if (i < K) {
            const int32_t h = v - (n - hub_cap);
            din = indeg[h];
            ri = rowinfo[v];
            e0 = hub_start[h];
            // the scatter must have filled the hub's segment: a count and a scatter that
            // disagree are reported instead of trusted.  A shard's sources fill its front.
            const unsigned long long filled = cur[h] - (unsigned long long)e0;
            if (shard ? filled > din : filled != din) atomicOr(&stats->err, ERR_OVERFLOW);
            if (din > 0 && ri.y > 0) {
                big = din >= (uint32_t)big_in || ri.y > HUB_WARP_MAX;
                dwin = v >= T0w ? ri.y : (col[ri.x + ri.y - 1] >= T0w ? (int)winrow[v].y : 0);
                dlow = ri.y - dwin;
            }
            if (shard) din = (uint32_t)min(filled, (unsigned long long)din);
        }
        const bool lng = big && dlow > HUB_LIST_MIN;
        const unsigned pb = warp_append(big, &stats->hub_big);
        const unsigned pl = warp_append(lng, &stats->hub_long);
        if (big) big_list[pb] = v;
        if (lng) long_list[pl] = v;
        const unsigned ns = (din + HUB_SLICE - 1) / HUB_SLICE;
        const unsigned tb = warp_reserve(big && dwin > 0 ? ns : 0u, &stats->hub_tasks);
        const unsigned tm = warp_reserve(!big && dwin > 0 ? ns : 0u, &stats->hub_med);
        const unsigned tl = warp_reserve(dlow > 0 ? ns : 0u, &stats->hub_low);
        for (unsigned k = 0; k < ns && dlow + dwin > 0; ++k) {
            const int64_t slot = big ? (int64_t)tb + k : task_cap - 1 - (int64_t)tm - k;
            const uint32_t ne = min(din - k * HUB_SLICE, (uint32_t)HUB_SLICE);
            const int first = (int)(e0 + (int64_t)k * HUB_SLICE);
            if ((dwin > 0 && (slot < 0 || slot >= task_cap)) || (dlow > 0 && (int64_t)tl + k >= task_cap)) {
                atomicOr(&stats->err, ERR_OVERFLOW);  // never: hub_task_cap
                break;
            }
            if (dwin > 0) win_task[slot] = make_int4(v, first, ri.x + dlow, (int)(ne | (uint32_t)dwin << TASK_BITS));
            if (dlow > 0) low_task[tl + k] = make_int4(v, first, (int)ne, dlow);
        }
    }
}

// Push lists: sources with at least one non-hub target and a non-empty suffix.  A
// block classifies PLAN_ITEMS vertices per thread and appends them with one global
// atomic per list and block (warp ballots, then shared-memory offsets), since one
// atomic per warp and list serialises on the four list counters.
constexpr int PLAN_ITEMS = 4;
constexpr int PLAN_LISTS = 5;  // d+ classes <= 8, <= 16, <= 32, <= SMALL_WIDE_MAX, larger
static_assert(PUSH_LIST_MIN[0] == 2 && PUSH_LIST_MIN[1] == 9 && PUSH_LIST_MIN[2] == 17 && PUSH_LIST_MIN[3] == 33 &&
                  PUSH_LIST_MIN[4] == SMALL_WIDE_MAX + 1,
              "a class's least d+ bounds its list");

// How often the probes of the hub kernels hit, from rows spread over the ranks: is the entry
// in the middle of a row's upper half in the list of the one in the row's middle, a hub?
// Where more than half are, the graph is one of communities (hub_dense).  R-MAT graphs of
// 2^12 .. 2^23 vertices have 0.23 .. 0.03, uniform ones next to none, geometric ones 0.7,
// disjoint cliques 1.  The first blocks of k_plan do this beside the others' work.
constexpr int SAMPLE_BLOCKS_MAX = 64;
constexpr int sample_blocks(int32_t n) {
    return n >= SAMPLE_BLOCKS_MAX * 1024 ? SAMPLE_BLOCKS_MAX : (n + 1023) / 1024;
}
__device__ __forceinline__ void sample_hubs(int32_t n, int32_t R, int blocks, const int2* __restrict__ rowinfo,
                                            const int32_t* __restrict__ col, DevStats* stats) {
    const int64_t i = (int64_t)blockIdx.x * THREADS + threadIdx.x, all = (int64_t)blocks * THREADS;
    const int2 ru = rowinfo[i * n / all];
    bool sampled = false, hit = false;
    if (ru.y >= 2) {
        const int mid = (ru.y - 1) / 2;  // before the last entry
        const int32_t v = col[ru.x + mid], x = col[ru.x + mid + (ru.y - mid) / 2];
        sampled = v >= R;
        if (sampled) {
            const int2 rv = rowinfo[v];
            const int p = lower_bound(col + rv.x, 0, rv.y, x);
            hit = p < rv.y && col[rv.x + p] == x;
        }
    }
    const unsigned sm = __ballot_sync(FULL, sampled), hm = __ballot_sync(FULL, hit);
    if (lane_id() == 0 && sm) {
        atomicAdd(&stats->samples, (unsigned)__popc(sm));
        if (hm) atomicAdd(&stats->sample_hits, (unsigned)__popc(hm));
    }
}
__device__ __forceinline__ bool hub_dense(const DevStats* stats) { return 2 * stats->sample_hits > stats->samples; }

__global__ void __launch_bounds__(THREADS) k_plan(int32_t n, int samplers, const int64_t* __restrict__ rowstart,
                                                  const int32_t* __restrict__ rowlen,
                                                  const int2* __restrict__ rowinfo, const int32_t* __restrict__ col,
                                                  int32_t* __restrict__ l8, int32_t* __restrict__ l16,
                                                  int32_t* __restrict__ l32, int32_t* __restrict__ l256,
                                                  int32_t* __restrict__ lcta, int32_t src_lo, int32_t src_hi,
                                                  DevStats* stats) {
    __shared__ unsigned bcount[PLAN_LISTS];
    __shared__ unsigned bbase[PLAN_LISTS];
    const int32_t R = n - (int32_t)stats->hub_count;
    const int lane = lane_id();
    unsigned* counters[PLAN_LISTS] = {&stats->small_count[0], &stats->small_count[1], &stats->small_count[2],
                                      &stats->small_count[3], &stats->cta_count};
    int32_t* lists[PLAN_LISTS] = {l8, l16, l32, l256, lcta};
    if ((int)blockIdx.x < samplers) {
        if (R < n) sample_hubs(n, R, samplers, rowinfo, col, stats);
        return;
    }
    const int64_t tile = (int64_t)THREADS * PLAN_ITEMS;
    for (int64_t t0 = (int64_t)(blockIdx.x - samplers) * tile; t0 < n; t0 += (int64_t)(gridDim.x - samplers) * tile) {
        if (threadIdx.x < PLAN_LISTS) bcount[threadIdx.x] = 0;
        __syncthreads();
        int cls[PLAN_ITEMS];
        unsigned off[PLAN_ITEMS];
#pragma unroll
        for (int k = 0; k < PLAN_ITEMS; ++k) {
            const int64_t u = t0 + (int64_t)k * THREADS + threadIdx.x;
            int d = u < n && u >= src_lo && u < src_hi ? rowlen[u] : 0;  // sources outside the shard: none
            if (d >= 2 && col[rowstart[u]] >= R) d = 0;  // every target is a hub
            cls[k] = d < 2 ? -1 : d <= 8 ? 0 : d <= 16 ? 1 : d <= 32 ? 2 : d <= SMALL_WIDE_MAX ? 3 : 4;
#pragma unroll
            for (int c = 0; c < PLAN_LISTS; ++c) {
                const unsigned mk = __ballot_sync(FULL, cls[k] == c);
                unsigned wb = 0;
                if (mk && lane == 0) wb = atomicAdd(&bcount[c], (unsigned)__popc(mk));
                wb = __shfl_sync(FULL, wb, 0);
                if (cls[k] == c) off[k] = wb + __popc(mk & lanemask_lt());
            }
        }
        __syncthreads();
        if (threadIdx.x < PLAN_LISTS)
            bbase[threadIdx.x] = bcount[threadIdx.x] ? atomicAdd(counters[threadIdx.x], bcount[threadIdx.x]) : 0u;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < PLAN_ITEMS; ++k)
            if (cls[k] >= 0) lists[cls[k]][bbase[cls[k]] + off[k]] = (int32_t)(t0 + (int64_t)k * THREADS + threadIdx.x);
        __syncthreads();
    }
}

// ---- small bucket: groups of G lanes, one lane per edge -----------------------

template <int G>
__global__ void __launch_bounds__(SMALL_WARPS * 32, SMALL_BLOCKS) k_tc_small(int32_t n, const int64_t* __restrict__ rowstart,
                                                               const int32_t* __restrict__ rowlen,
                                                               const int2* __restrict__ rowinfo,
                                                               const int32_t* __restrict__ col,
                                                               const int32_t* __restrict__ list, int cls,
                                                               unsigned long long* __restrict__ t, DevStats* stats,
                                                               int strategy, float factor) {
    constexpr int GPW = 32 / G;
    __shared__ int32_t sLu[SMALL_WARPS * 32];
    __shared__ uint32_t sCnt[SMALL_WARPS * 32];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int grp = lane / G, g = lane % G;
    const unsigned gmask = G == 32 ? FULL : (((1u << G) - 1u) << (grp * G));
    int32_t* Lu = sLu + w * 32 + grp * G;
    uint32_t* cnt = sCnt + w * 32 + grp * G;
    const unsigned count = stats->small_count[cls];
    const int32_t R = n - (int32_t)stats->hub_count;
    const unsigned groups = gridDim.x * SMALL_WARPS * GPW;
    // the next source and its row are fetched while the current one is counted
    unsigned q = (blockIdx.x * SMALL_WARPS + w) * GPW + grp;
    int32_t u = q < count ? list[q] : 0;
    int2 ru = q < count ? rowinfo[u] : make_int2(0, 0);
    for (; q < count; q += groups) {
        const unsigned qn = q + groups;
        const int32_t un = qn < count ? list[qn] : 0;
        const int du = ru.y;
        const int64_t base = ru.x;
        Lu[g] = g < du ? col[base + g] : INT_MAX;
        cnt[g] = 0;
        const int2 run = qn < count ? rowinfo[un] : make_int2(0, 0);
        __syncwarp(gmask);
        uint32_t c = 0;
        if (g < du - 1) {
            const int32_t v = Lu[g];
            const int2 ri = v < R ? rowinfo[v] : make_int2(0, 0);
            const int dv = ri.y;
            if (dv > 0) {
                const int32_t* B = col + ri.x;
                const int a = du - g - 1;
                int method = strategy;
                if (method == TC_STRAT_AUTO) method = small_auto(a, dv, factor);
                if (method == TC_STRAT_MERGE)
                    c = lane_merge_batched(Lu, g + 1, du, B, dv, cnt);
                else
                    c = a <= dv ? lane_search(Lu, g + 1, du, B, dv, cnt)
                                : lane_search_rev(Lu, g + 1, du, B, dv, cnt);
                if (c) atomicAdd(&cnt[g], c);
            }
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) c += __shfl_down_sync(gmask, c, o, G);
        __syncwarp(gmask);
        const uint32_t cv = cnt[g];
        if (g < du && cv) atomicAdd(&t[Lu[g]], (unsigned long long)cv);
        if (g == 0 && c) atomicAdd(&t[u], (unsigned long long)c);
        __syncwarp(gmask);
        u = un;
        ru = run;
    }
}

// Sources with 32 < |N+(u)| <= SMALL_WIDE_MAX: a group of SMALL_WIDE_G lanes per
// source stages N+(u) in shared memory and its lanes take the edges (u, v) with v a
// non-hub (the first jh entries), one at a time, with the same per-edge choice
// (Eq. 3) between the batched merge and binary search as the small kernel.  Such
// sources mostly point to hubs and have few non-hub edges, so a block (or a whole
// warp) per source would idle.
constexpr int SMALL_WIDE_G = 16;
constexpr int SMALL_WIDE_BLOCKS = 6;  // blocks per SM
constexpr int SMALL_WIDE_GROUPS = SMALL_WARPS * 32 / SMALL_WIDE_G;  // per block

__global__ void __launch_bounds__(SMALL_WARPS * 32) k_tc_small_wide(int32_t n, const int2* __restrict__ rowinfo,
                                                                   const int32_t* __restrict__ col,
                                                                   const int32_t* __restrict__ list,
                                                                   unsigned long long* __restrict__ t,
                                                                   DevStats* stats, int strategy, float factor) {
    extern __shared__ __align__(16) unsigned char wide_sh[];
    constexpr int G = SMALL_WIDE_G;
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int grp = lane / G, g = lane % G;
    const unsigned gmask = G == 32 ? FULL : (((1u << G) - 1u) << (grp * G));
    const int gi = w * (32 / G) + grp;  // group index in the block
    int32_t* Lu = reinterpret_cast<int32_t*>(wide_sh) + gi * SMALL_WIDE_MAX;
    uint32_t* cnt = reinterpret_cast<uint32_t*>(wide_sh) + (SMALL_WIDE_GROUPS + gi) * SMALL_WIDE_MAX;
    const unsigned count = stats->small_count[3];
    const int32_t R = n - (int32_t)stats->hub_count;
    const unsigned groups = gridDim.x * SMALL_WIDE_GROUPS;
    for (unsigned q = blockIdx.x * SMALL_WIDE_GROUPS + gi; q < count; q += groups) {
        const int32_t u = list[q];
        const int2 ru = rowinfo[u];
        const int du = ru.y;  // 33 .. SMALL_WIDE_MAX
        for (int p = g; p < du; p += G) {
            Lu[p] = col[ru.x + p];
            cnt[p] = 0;
        }
        __syncwarp(gmask);
        const int jh = min(du - 1, lower_bound(Lu, 0, du, R));  // edges into non-hubs
        uint32_t c = 0;
        for (int j = g; j < jh; j += G) {
            const int32_t v = Lu[j];
            const int2 ri = rowinfo[v];
            const int dv = ri.y;
            if (dv == 0) continue;
            const int32_t* B = col + ri.x;
            const int a = du - j - 1;
            int method = strategy;
            if (method == TC_STRAT_AUTO) method = small_auto(a, dv, factor);
            const uint32_t cj = method == TC_STRAT_MERGE
                                    ? lane_merge_batched(Lu, j + 1, du, B, dv, cnt)
                                    : (a <= dv ? lane_search(Lu, j + 1, du, B, dv, cnt)
                                               : lane_search_rev(Lu, j + 1, du, B, dv, cnt));
            if (cj) atomicAdd(&cnt[j], cj);
            c += cj;
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) c += __shfl_down_sync(gmask, c, o, G);
        __syncwarp(gmask);
        for (int p = g; p < du; p += G) {
            const uint32_t cv = cnt[p];
            if (cv) atomicAdd(&t[Lu[p]], (unsigned long long)cv);
        }
        if (g == 0 && c) atomicAdd(&t[u], (unsigned long long)c);
        __syncwarp(gmask);
    }
}

// ---- block bucket: |N+(u)| > 256, non-hub targets ------------------------------

// Open-addressing hash set of a staged list in shared memory (Fibonacci hashing, linear
// probing, empty slots hold -1).  The table has at least twice as many slots as
// keys, so a probe meets an empty slot after about two steps at most on average.
struct HashProbe {
    const int32_t* keys;
    unsigned shift, mask;
    __device__ __forceinline__ int operator()(int32_t x) const {
        unsigned h = ((unsigned)x * 0x9e3779b1u) >> shift;
        for (;;) {
            const int32_t k = keys[h];
            if (k == x) return (int)h;
            if (k < 0) return -1;
            h = (h + 1) & mask;
        }
    }
};

// 1 << d for d in [0, 32), 0 for any other d (PTX clamps the shift amount).
__device__ __forceinline__ unsigned bit_or_none(int d) {
    unsigned r;
    asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(d));
    return r;
}

// Inclusive warp scan whose adds are predicated by the shuffles themselves.  Volatile: all
// lanes take part, so no step may be merged with another or sink into a branch.
__device__ __forceinline__ uint32_t warp_scan_u32(uint32_t x) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
        asm volatile("{ .reg .pred p; .reg .u32 y; shfl.sync.up.b32 y|p, %0, %1, 0, 0xffffffff; @p add.u32 %0, %0, y; }"
            : "+r"(x)
            : "r"(o));
    return x;
}

// One warp's edges (up to 32) with something to read, in order: lane i takes the i-th of
// them.  Their items are laid end to end; at[i] = {base of edge i's items less the
// items before it, their end}.
struct EdgeItems {
    int cz, total, excl;  // edges; items; first item of this lane's edge (-1: none)
    int seen;             // edges that start before the round, less one
    unsigned upto;        // this lane's bit and those below it

    // items: this lane's edge's count; returns the lane whose edge this lane takes
    __device__ __forceinline__ int gather(int items, uint32_t* cw) {
        const int lane = lane_id();
        const unsigned nz = __ballot_sync(FULL, items > 0);
        cz = __popc(nz);
        if (cz == 0) return 0;
        if (items > 0) cw[__popc(nz & lanemask_lt())] = (uint32_t)lane;
        __syncwarp();
        return lane < cz ? (int)cw[lane] : lane;
    }
    // items and base of the edge this lane has taken
    __device__ __forceinline__ void lay(int items, int base, int2* at) {
        const int lane = lane_id();
        if (lane >= cz) items = 0;
        const int incl = (int)warp_scan_u32((uint32_t)items);
        total = __shfl_sync(FULL, incl, 31);
        excl = lane < cz ? incl - items : -1;
        at[lane] = make_int2(base - (incl - items), incl);
        seen = -1;
        upto = lane == 31 ? FULL : (2u << lane) - 1u;
        __syncwarp();
    }
    // the edge of item r + lane; called for r = 0, 32, 64, ... in turn
    __device__ __forceinline__ int edge_of(int r) {
        const unsigned mk = __reduce_or_sync(FULL, bit_or_none(excl - r));
        const int i = seen + __popc(mk & upto);
        seen += __popc(mk);
        return i;
    }
};

// ---- small bucket, hash strategy: N+(u) as a hash set, target rows end to end ----

// Open-addressing set whose slots say in bit 31 whether an insertion went past them: a
// probe of any other key ends at the first unmarked slot, whatever key it holds (at a
// quarter of the slots taken, one probe in a hundred goes on; without the marks every
// fourth).  Ranks are below 2^31 - 1, which marks an empty slot.
constexpr int32_t SET_EMPTY = INT_MAX;

template <int LG>
struct MarkedSet {
    int32_t* keys;
    static __device__ __forceinline__ unsigned slot(int32_t x) { return ((unsigned)x * 0x9e3779b1u) >> (32 - LG); }
    static __device__ __forceinline__ unsigned after(unsigned h) { return (h + 1) & ((1u << LG) - 1u); }
    __device__ __forceinline__ unsigned insert(int32_t x) const {  // keys are distinct
        unsigned h = slot(x);
        while (atomicCAS(&keys[h], SET_EMPTY, x) != SET_EMPTY) {
            atomicOr(&keys[h], INT_MIN);
            h = after(h);
        }
        return h;
    }
    __device__ __forceinline__ int operator()(int32_t x) const {
        unsigned h = slot(x);
        for (;;) {
            const int32_t k = keys[h];
            if ((k & INT_MAX) == x) return (int)h;
            if (k >= 0) return -1;
            h = after(h);
        }
    }
};

// A warp takes one source u at a time.  N+(u) (at most SL / 2 entries) goes into a set of
// SL slots in shared memory.  Its edges (u, v) into non-hubs are taken 32 at a time; their
// rows N+(v) are laid end to end and read 32 entries per round, one per lane, each probed
// once (entries above max N+(u) are skipped).  A hit at x in N+(v) is a triangle: x is
// above v, so it lies in the suffix of N+(u) after v, which is W for the edge (u, v).
// Hits add to the slot's counter (t[x], flushed once per source); at an edge's last entry
// the hits up to it are noted, so that differences give each edge's count (t[v]); their
// sum goes to t[u].
//
// Bound by instruction issue (75 to 78 % of the slots; 27 of 32 lanes active).  A batch of
// 840 graphs, 66 M pairs, sources of 17..32 and 33..256 entries: one edge at a time with
// whole warps, 2.0 and 3.3 ms; rows end to end, 1.3 and 3.0; with sources claimed one by
// one (a static stride left the last warps 20 % longer), 1.1 and 2.5.  4, 5, 7 and 8 blocks
// per SM are 2 to 25 % slower than 6.
constexpr int HASH_BLOCKS = 6;  // resident blocks per SM: the grid is one wave of them
template <int LG, bool SUP>
__global__ void __launch_bounds__(SMALL_WARPS * 32, SUP ? 4 : HASH_BLOCKS)
    k_tc_small_hash(int32_t n, const int2* __restrict__ rowinfo, const int32_t* __restrict__ col,
                    const int32_t* __restrict__ list, int cls, unsigned long long* __restrict__ t, DevStats* stats,
                    uint32_t* __restrict__ sup_arg) {
    uint32_t* const sup = SUP ? sup_arg : nullptr;
    constexpr int SL = 1 << LG;
    __shared__ int32_t skeys[SMALL_WARPS][SL];
    __shared__ uint32_t shcnt[SMALL_WARPS][SL];
    __shared__ uint16_t shpos[SMALL_WARPS][SUP ? SL : 1];  // position in N+(u) of each key (support only)
    __shared__ int2 sat[SMALL_WARPS][32];
    __shared__ uint32_t scw[SMALL_WARPS][32];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const MarkedSet<LG> P{skeys[w]};
    uint32_t* const hcnt = shcnt[w];
    uint16_t* const hpos = shpos[w];
    int2* const at = sat[w];
    uint32_t* const cw = scw[w];
    for (int i = lane; i < SL; i += 32) {
        P.keys[i] = SET_EMPTY;
        hcnt[i] = 0;
    }
    __syncwarp();
    const unsigned count = stats->small_count[cls];
    const int32_t R = n - (int32_t)stats->hub_count;
    // sources are claimed one ahead, and the next one's row is fetched meanwhile
    unsigned q = blockIdx.x * SMALL_WARPS + w;
    int32_t u = q < count ? list[q] : 0;
    int2 ru = q < count ? rowinfo[u] : make_int2(0, 0);
    while (q < count) {
        unsigned qn = 0;
        if (lane == 0) qn = gridDim.x * SMALL_WARPS + atomicAdd(&stats->small_next[cls - 2], 1u);
        qn = __shfl_sync(FULL, qn, 0);
        const int32_t un = qn < count ? list[qn] : 0;
        const int du = ru.y;
        const int64_t base = ru.x;
        int jh = 0;  // entries below the hubs: the rows are sorted, so they come first
        for (int i0 = 0; i0 < du; i0 += 32) {
            const bool valid = i0 + lane < du;
            const int32_t x = valid ? col[base + i0 + lane] : INT_MAX;
            if (valid) {
                const unsigned h = P.insert(x);
                if (sup) hpos[h] = (uint16_t)(i0 + lane);
            }
            jh += __popc(__ballot_sync(FULL, x < R));
        }
        const int32_t maxu = col[base + du - 1];
        const int2 run = qn < count ? rowinfo[un] : make_int2(0, 0);
        const int ne = min(jh, du - 1);  // the last entry has an empty suffix
        __syncwarp();
        uint32_t cu = 0;
        for (int e0 = 0; e0 < ne; e0 += 32) {
            const bool has = e0 + lane < ne;
            const int32_t v0 = has ? col[base + e0 + lane] : 0;
            const int2 r0 = has ? rowinfo[v0] : make_int2(0, 0);
            // only entries up to max N+(u) can match: long rows are cut there; an edge
            // whose cut row is longer than the suffix a of N+(u) after v by more than
            // Eq. 3 allows (factor 8: one lane's dependent search steps cost more than the
            // warp's parallel probes) is left to its own lane, which searches the a keys
            // in the row (a log b instead of b probes)
            int b = r0.y;
            if (b > HASH_CUT) b = lower_bound(col + r0.x, 0, b, maxu + 1);
            const int a = du - (e0 + lane) - 1;
            const bool search = b > 0 && a > 0 && b > a && !eq3_prefers_merge(a, b, 8.0f);
            uint32_t cs = 0;  // a searching lane: the suffix keys after v looked up in N+(v)
            if (search) {
                const int32_t* B = col + r0.x;
                int lo = 0;
                for (int i = e0 + lane + 1; i < du && lo < b; ++i) {
                    const int32_t y = col[base + i];
                    const int p = lower_bound(B, lo, b, y);
                    lo = p;
                    if (p < b && B[p] == y) {
                        atomicAdd(&hcnt[P(y)], 1u);
                        if (sup) atomicAdd(&sup[r0.x + p], 1u);  // edge (v, y)
                        ++cs;
                    }
                }
                if (cs) {
                    atomicAdd(&t[v0], (unsigned long long)cs);
                    if (sup) atomicAdd(&sup[base + e0 + lane], cs);  // edge (u, v)
                }
            }
            __syncwarp();
            cu += cs;
            EdgeItems E;
            const int src = E.gather(search ? 0 : b, cw);
            if (E.cz == 0) continue;
            const int32_t v = __shfl_sync(FULL, v0, src);
            E.lay(__shfl_sync(FULL, b, src), __shfl_sync(FULL, r0.x, src), at);
            uint32_t running = 0;
            for (int r = 0; r < E.total; r += 64) {
                const int item = r + lane;
                int idx[2];
                int2 e[2];
                int32_t x[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    idx[h] = 0;
                    e[h] = make_int2(0, 0);
                    x[h] = INT_MAX;
                    if (h == 0 || r + 32 < E.total) {
                        idx[h] = E.edge_of(r + 32 * h);
                        e[h] = at[idx[h]];
                        if (item + 32 * h < E.total) x[h] = col[e[h].x + item + 32 * h];
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int slot = x[h] <= maxu ? P(x[h]) : -1;
                    if (slot >= 0) {
                        atomicAdd(&hcnt[slot], 1u);
                        if (sup) atomicAdd(&sup[e[h].x + item + 32 * h], 1u);  // edge (v, x)
                    }
                    const unsigned hits = __ballot_sync(FULL, slot >= 0);
                    // an edge's last entry
                    if (e[h].y == item + 32 * h + 1) cw[idx[h]] = running + __popc(hits & E.upto);
                    running += __popc(hits);
                }
            }
            __syncwarp();
            if (lane < E.cz) {
                const uint32_t ce = cw[lane] - (lane ? cw[lane - 1] : 0u);
                if (ce) {
                    atomicAdd(&t[v], (unsigned long long)ce);
                    if (sup) atomicAdd(&sup[base + e0 + src], ce);  // edge (u, v)
                    cu += ce;
                }
            }
            __syncwarp();
        }
        cu = __reduce_add_sync(FULL, cu);
        if (lane == 0 && cu) atomicAdd(&t[u], (unsigned long long)cu);
        for (int i = lane; i < SL; i += 32) {  // flush the per-entry counts, empty the set
            const int32_t x = P.keys[i] & INT_MAX;
            if (x != SET_EMPTY) {
                const uint32_t c = hcnt[i];
                if (c) {
                    atomicAdd(&t[x], (unsigned long long)c);
                    if (sup) atomicAdd(&sup[base + hpos[i]], c);  // edge (u, x)
                }
                P.keys[i] = SET_EMPTY;
                hcnt[i] = 0;
            }
        }
        __syncwarp();
        q = qn;
        u = un;
        ru = run;
    }
}

// Sources of at most G = 8 or 16 entries, 32 / G of them by a warp: each lane has one entry
// of one source, inserts it into that source's set of 4 G slots and keeps its slot.  The
// edges of all of them go end to end as above; a hit adds to the slot's counter and to the
// edge's, kept with the lane that has the entry, which so flushes t[x] and the edge's
// support once.
//
// Bound by the random sectors of row records and rows: a uniform graph of 2^23 vertices and
// 60 M pairs, sources of up to 8 and 9..16 entries: a merge per lane, 10 to 12 lanes of 32
// active, 0.66 and 1.20 ms; this, 0.47 and 0.75 (the second reads 3.8 GB).  A batch of 840
// graphs, 66 M pairs: 0.43 and 0.90, now 0.48 and 0.76.  6 blocks per SM (37 registers)
// instead of 8 take 10 to 20 % longer.
constexpr int SETS_LONG = 32;   // Eq. 3 (factor 8) searches no row of at most so many entries
constexpr int SETS_BLOCKS = 8;  // resident blocks per SM: the grid is one wave of them
template <int G, bool SUP>
__global__ void __launch_bounds__(SMALL_WARPS * 32, SETS_BLOCKS)
    k_tc_small_sets(int32_t n, const int2* __restrict__ rowinfo, const int32_t* __restrict__ col,
                    const int32_t* __restrict__ list, int cls, unsigned long long* __restrict__ t, DevStats* stats,
                    uint32_t* __restrict__ sup_arg) {
    uint32_t* const sup = SUP ? sup_arg : nullptr;
    constexpr int GPW = 32 / G, SL = 4 * G;
    using Set = MarkedSet<G == 8 ? 5 : 6>;
    static_assert(SL == (G == 8 ? 32 : 64), "slots of a set");
    __shared__ int32_t skeys[SMALL_WARPS][GPW * SL];
    __shared__ uint32_t shcnt[SMALL_WARPS][GPW * SL];
    __shared__ int2 sat[SMALL_WARPS][32];
    __shared__ uint32_t sce[SMALL_WARPS][32];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int grp = lane / G, gl = lane % G;
    int32_t* const keys = skeys[w];
    uint32_t* const hcnt = shcnt[w];
    int2* const at = sat[w];
    uint32_t* const ce = sce[w];
    for (int i = lane; i < GPW * SL; i += 32) {
        keys[i] = SET_EMPTY;
        hcnt[i] = 0;
    }
    __syncwarp();
    const Set own{keys + grp * SL};
    const unsigned count = stats->small_count[cls];
    const int32_t R = n - (int32_t)stats->hub_count;
    const unsigned step = gridDim.x * SMALL_WARPS * GPW;
    unsigned q0 = (blockIdx.x * SMALL_WARPS + w) * GPW;  // the warp's first source
    int32_t u = q0 + grp < count ? list[q0 + grp] : 0;
    int2 ru = q0 + grp < count ? rowinfo[u] : make_int2(0, 0);
    int32_t x = gl < ru.y ? col[ru.x + gl] : INT_MAX;
    for (; q0 < count; q0 += step) {
        const unsigned qn = q0 + step + grp;  // the next source and its row are fetched ahead
        const int32_t un = qn < count ? list[qn] : 0;
        const int du = ru.y;
        const bool has = gl < du;
        const int2 rx = gl < du - 1 && x < R ? rowinfo[x] : make_int2(0, 0);  // the last entry has an empty suffix
        const int2 run = qn < count ? rowinfo[un] : make_int2(0, 0);
        unsigned hs = grp * SL;
        if (has) hs += own.insert(x);
        __syncwarp();
        uint32_t cs = 0;
        int b = rx.y;
        if (__any_sync(FULL, b > SETS_LONG)) {  // long rows: as in k_tc_small_hash
            const int32_t maxu = __shfl_sync(FULL, x, grp * G + (du > 0 ? du - 1 : 0));
            if (b > HASH_CUT) b = lower_bound(col + rx.x, 0, b, maxu + 1);
            const int a = du - gl - 1;
            if (b > SETS_LONG && !eq3_prefers_merge(a, b, 8.0f)) {
                const int32_t* B = col + rx.x;
                int lo = 0;
                for (int i = gl + 1; i < du && lo < b; ++i) {
                    const int32_t y = col[ru.x + i];
                    const int p = lower_bound(B, lo, b, y);
                    lo = p;
                    if (p < b && B[p] == y) {
                        atomicAdd(&hcnt[grp * SL + own(y)], 1u);
                        if (sup) atomicAdd(&sup[rx.x + p], 1u);  // edge (v, y)
                        ++cs;
                    }
                }
                b = 0;
            }
        }
        __syncwarp();
        const int32_t xn = gl < run.y ? col[run.x + gl] : INT_MAX;
        EdgeItems E;
        const int src = E.gather(b, ce);
        if (E.cz) {
            E.lay(__shfl_sync(FULL, b, src), __shfl_sync(FULL, rx.x, src), at);
            if (lane < E.cz) at[lane].y = src;
            ce[lane] = 0;
            __syncwarp();
            for (int r = 0; r < E.total; r += 64) {
                const int item = r + lane;
                int2 e[2];
                int32_t y[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    e[h] = make_int2(0, 0);
                    y[h] = INT_MAX;
                    if (h == 0 || r + 32 < E.total) {
                        e[h] = at[E.edge_of(r + 32 * h)];
                        if (item + 32 * h < E.total) y[h] = col[e[h].x + item + 32 * h];
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int set = (e[h].y & ~(G - 1)) * (SL / G);
                    const int slot = y[h] != INT_MAX ? Set{keys + set}(y[h]) : -1;
                    if (slot >= 0) {
                        atomicAdd(&hcnt[set + slot], 1u);
                        atomicAdd(&ce[e[h].y], 1u);
                        if (sup) atomicAdd(&sup[e[h].x + item + 32 * h], 1u);  // edge (v, y)
                    }
                }
            }
            __syncwarp();
            cs += ce[lane];
        }
        uint32_t cu = cs;
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) cu += __shfl_xor_sync(FULL, cu, o);
        if (has) {  // flush the entry's counts, empty its slot
            const uint32_t cx = hcnt[hs] + cs;
            if (cx) {
                atomicAdd(&t[x], (unsigned long long)cx);
                if (sup) atomicAdd(&sup[ru.x + gl], cx);  // edge (u, x): as v of its edge and as w of others
            }
            keys[hs] = SET_EMPTY;
            hcnt[hs] = 0;
        }
        if (gl == 0 && cu) atomicAdd(&t[u], (unsigned long long)cu);
        __syncwarp();
        u = un;
        ru = run;
        x = xn;
    }
}

// Warp per edge: the entries of B = N+(v) (sorted) are probed in a set of the
// staged N+(u), two per lane per round, stopping above max N+(u); hits add to the
// set's per-slot counter.  Returns the edge's count (all lanes).
template <class Probe>
__device__ uint32_t edge_probe_set(const Probe& P, int32_t maxu, uint32_t* hcnt, const int32_t* __restrict__ B, int b,
                               uint32_t* __restrict__ supB) {
    const int lane = lane_id();
    uint32_t c = 0;
    for (int k0 = 0; k0 < b; k0 += 64) {
        const int k1 = k0 + lane, k2 = k1 + 32;
        const int32_t x1 = k1 < b ? B[k1] : INT_MAX;
        const int32_t x2 = k2 < b ? B[k2] : INT_MAX;
        if (x1 <= maxu) {
            const int p = P(x1);
            if (p >= 0) {
                atomicAdd(&hcnt[p], 1u);
                if (supB) atomicAdd(&supB[k1], 1u);
                ++c;
            }
        }
        if (x2 <= maxu) {
            const int p = P(x2);
            if (p >= 0) {
                atomicAdd(&hcnt[p], 1u);
                if (supB) atomicAdd(&supB[k2], 1u);
                ++c;
            }
        }
        if (__any_sync(FULL, x2 > maxu)) break;  // B is sorted
    }
    return warp_sum(c);
}

struct CtaShared {
    int32_t Lu[CTA_LIST_MAX];
    uint32_t cnt[CTA_LIST_MAX];
    union {
        struct {  // bitmap of N+(u) over its rank window
            uint32_t bm[BITMAP_WORDS];
            uint16_t pre[BITMAP_WORDS];
            uint32_t slice[BITMAP_WORDS / 32];
        } b;
        struct {  // hash set of N+(u) when the window is wider than the bitmap
            int32_t keys[2 * CTA_LIST_MAX];
            uint32_t hcnt[2 * CTA_LIST_MAX];
        } h;
    } s;
    unsigned long long utot[CTA_WARPS];
    int q;
};

template <bool SUP>
__global__ void __launch_bounds__(CTA_THREADS) k_tc_cta(int32_t n, const int64_t* __restrict__ rowstart,
                                                        const int32_t* __restrict__ rowlen,
                                                        const int2* __restrict__ rowinfo,
                                                        const int32_t* __restrict__ col,
                                                        const int32_t* __restrict__ list,
                                                        unsigned long long* __restrict__ t,
                                                        DevStats* stats, int strategy, float factor,
                                                        uint32_t* __restrict__ sup_arg) {
    uint32_t* const sup = SUP ? sup_arg : nullptr;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    CtaShared& sh = *reinterpret_cast<CtaShared*>(smem_raw);
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const unsigned count = stats->cta_count;
    const int32_t R = n - (int32_t)stats->hub_count;
    for (;;) {
        if (threadIdx.x == 0) sh.q = (int)atomicAdd(&stats->cta_next, 1u);
        __syncthreads();
        const int q = sh.q;
        if ((unsigned)q >= count) break;
        const int32_t u = list[q];
        const int du = rowlen[u];
        const int64_t base = rowstart[u];
        const bool staged = du <= CTA_LIST_MAX;
        if (staged) {
            for (int p = threadIdx.x; p < du; p += CTA_THREADS) {
                sh.Lu[p] = col[base + p];
                sh.cnt[p] = 0;
            }
        }
        __syncthreads();
        const int32_t* Lu = staged ? sh.Lu : col + base;
        const int32_t maxu = Lu[du - 1];
        const int jh = min(du - 1, lower_bound(Lu, 0, du, R));  // edges into non-hubs
        const int span = maxu - u;  // ranks u+1 .. maxu
        const bool bitmap = staged && strategy == TC_STRAT_BITMAP && span <= BITMAP_WORDS * 32;
        const bool hashed = staged && strategy == TC_STRAT_BITMAP && !bitmap;
        if (bitmap) build_bitmap<CTA_THREADS>(sh.s.b.bm, sh.s.b.pre, sh.s.b.slice, sh.Lu, du, u, (span + 31) >> 5);
        unsigned hshift = 0, hmask = 0;
        if (hashed) {  // uniform across the block
            int lg = 6;
            while ((1 << lg) < 2 * du) ++lg;  // du <= CTA_LIST_MAX: at most 2 * CTA_LIST_MAX slots
            hmask = (1u << lg) - 1u;
            hshift = 32u - (unsigned)lg;
            for (int p = threadIdx.x; p <= (int)hmask; p += CTA_THREADS) {
                sh.s.h.keys[p] = -1;
                sh.s.h.hcnt[p] = 0;
            }
            __syncthreads();
            for (int p = threadIdx.x; p < du; p += CTA_THREADS) {
                const int32_t x = sh.Lu[p];
                unsigned h = ((unsigned)x * 0x9e3779b1u) >> hshift;
                while (atomicCAS(&sh.s.h.keys[h], -1, x) != -1) h = (h + 1) & hmask;  // keys are distinct
            }
            __syncthreads();
        }
        uint32_t* supA = sup ? sup + base : nullptr;
        Sink S{staged ? sh.cnt : nullptr, t, Lu, staged ? nullptr : supA, nullptr};
        unsigned long long utot = 0;
        for (int j = w; j < jh; j += CTA_WARPS) {
            const int32_t v = Lu[j];
            const int2 ri = rowinfo[v];
            const int dv = ri.y;
            if (dv == 0) continue;
            const int32_t* B = col + ri.x;
            uint32_t* supB = sup ? sup + ri.x : nullptr;
            S.supB = supB;
            uint32_t c;
            if (bitmap) {
                c = edge_bitmap(sh.s.b.bm, sh.s.b.pre, u, maxu, sh.cnt, B, dv, supB);
            } else if (hashed) {
                c = edge_probe_set(HashProbe{sh.s.h.keys, hshift, hmask}, maxu, sh.s.h.hcnt, B, dv, supB);
            } else {
                int method = strategy;
                if (method == TC_STRAT_AUTO) {
                    const int a = du - j - 1;
                    method = eq3_prefers_merge(a, dv, factor) ? TC_STRAT_MERGE
                                                              : (a <= dv ? TC_STRAT_SEARCH : TC_STRAT_PROBE);
                } else if (method == TC_STRAT_BITMAP) {
                    method = TC_STRAT_PROBE;
                }
                c = edge_dispatch(method, S, j + 1, du, B, dv);
            }
            if (lane == 0 && c) {
                if (staged) {
                    atomicAdd(&sh.cnt[j], c);
                } else {
                    atomicAdd(&t[v], (unsigned long long)c);
                    if (supA) atomicAdd(&supA[j], c);  // edge (u, v)
                }
            }
            utot += c;
        }
        if (lane == 0) sh.utot[w] = utot;
        __syncthreads();
        if (staged) {
            for (int p = threadIdx.x; p < du; p += CTA_THREADS) {
                const uint32_t cv = sh.cnt[p];
                if (cv) {
                    atomicAdd(&t[sh.Lu[p]], (unsigned long long)cv);
                    if (supA) atomicAdd(&supA[p], cv);
                }
            }
        }
        if (hashed) {
            for (int p = threadIdx.x; p <= (int)hmask; p += CTA_THREADS) {
                const int32_t x = sh.s.h.keys[p];
                const uint32_t cv = sh.s.h.hcnt[p];
                if (x >= 0 && cv) {
                    atomicAdd(&t[x], (unsigned long long)cv);
                    if (supA) atomicAdd(&supA[lower_bound(sh.Lu, 0, du, x)], cv);
                }
            }
        }
        if (threadIdx.x == 0) {
            unsigned long long s = 0;
            for (int k = 0; k < CTA_WARPS; ++k) s += sh.utot[k];
            if (s) atomicAdd(&t[u], s);
        }
        __syncthreads();
    }
}

// ---- hub bucket ----------------------------------------------------------------
// Every hub's in-edges stream their suffixes against the hub's staged list N+(v).  The
// windows of ranks (k_win_build) are counted apart: a suffix's entries in a window come
// eight to a load as offsets into what is staged of N+(v) there, so a probe is one
// shared-memory load.
//   k_tc_hub      window 1, big hubs (in-degree >= the planner's threshold, or lists too
//                 long for one warp): a block per slice of the in-edges
//   k_tc_hub_med  window 1, the other hubs: a warp per hub
//   k_tc_hub_win2 the windows below: a warp per slice
//   k_tc_hub_low  the same for per-edge support, over a hash set of 32-bit ids
//   k_tc_hub_list per-edge support of big hubs with many entries below window 1; in probe
//                 mode all big hubs
// For R-MAT scale 20 / 23 they take 1.03 / 4.7 ms together; 32-bit ids against one bitmap
// or hash set per hub took 1.28 / 5.94 ms.

struct BitmapProbe {
    const uint32_t* bm;
    const uint16_t* pre;
    int32_t v;
    __device__ __forceinline__ int operator()(int32_t x) const {
        const int off = x - v - 1;
        const uint32_t word = bm[off >> 5], bit = 1u << (off & 31);
        return (word & bit) ? (int)pre[off >> 5] + __popc(word & (bit - 1)) : -1;
    }
};

struct ListProbe {
    const int32_t* L;
    int d;
    __device__ __forceinline__ int operator()(int32_t x) const {
        const int p = lower_bound(L, 0, d, x);  // x <= max(L), so p < d
        return L[p] == x ? p : -1;
    }
};

// One batch of up to 32 in-edges [k0, min(k0 + 32, e1)) of hub v, processed by one warp
// over 32-bit ids (k_tc_hub_list): the whole suffixes, or (SUP) their entries below
// window 1.  Suffixes of HUB_LONG or more entries are read by lane groups (the read
// stops above max N+(v)); shorter ones are laid end to end and read 32 entries at a
// time.  Matches add to cnt[p] (or t[x] when cnt is null) and to the
// per-in-edge total, which goes to t[u].  Returns the batch total (all lanes).
template <bool SUP, class Probe>
__device__ uint32_t hub_batch(int64_t k0, int64_t e1, const uint2* __restrict__ in_rec,
                              const int2* __restrict__ rowinfo, const uint2* __restrict__ winrow,
                              const int32_t* __restrict__ col, int32_t maxv, const Probe& probe, uint32_t* cnt,
                              unsigned long long* __restrict__ t, uint32_t* cw, uint32_t* __restrict__ sup_arg,
                              int64_t vbase) {
    uint32_t* const sup = SUP ? sup_arg : nullptr;
    const int lane = lane_id();
    const int64_t k = k0 + lane;
    const uint2 rec = k < e1 ? in_rec[k] : make_uint2(0, 0);
    int32_t uu = (int32_t)rec.x;
    int32_t b0 = 0;
    int a = (int)rec.y;
    if (a > 0) {
        const int2 ri = rowinfo[uu];
        b0 = ri.x + ri.y - a;
        if (SUP) a -= (int)winrow[uu].y;
    }
    uint32_t total_c = 0;
    const bool islong = a >= HUB_LONG;
    const int nlong = __popc(__ballot_sync(FULL, islong));
    // the long suffixes by decreasing length (bitonic sort of (length, lane) keys across
    // the warp), so that the groups that run their rounds together take suffixes of
    // similar length and wait less for each other
    uint32_t key = islong ? ((uint32_t)min(a, (1 << 26) - 1) << 5) | (uint32_t)lane : 0u;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const uint32_t other = __shfl_xor_sync(FULL, key, j);
            const bool keep_max = ((lane & j) == 0) == ((lane & k) == 0);
            key = keep_max ? max(key, other) : min(key, other);
        }
    }
    // HUB_GROUPS long suffixes at a time, one per group of HUB_GLANES lanes, each lane
    // reading HUB_UNROLL entries per round with all loads in flight before any is used
    const int g = lane / HUB_GLANES, gl = lane % HUB_GLANES;
    const unsigned gmask = (HUB_GLANES == 32 ? FULL : ((1u << HUB_GLANES) - 1u)) << (g * HUB_GLANES);
    for (int k0 = 0; k0 < nlong; k0 += HUB_GROUPS) {
        const int pos = k0 + g;
        const uint32_t kp = __shfl_sync(FULL, key, min(pos, 31));
        const int my = pos < nlong ? (int)(kp & 31u) : -1;  // batch lane holding this group's in-edge
        const int src = my < 0 ? 0 : my;
        const int32_t bL = __shfl_sync(FULL, b0, src);
        int aL = __shfl_sync(FULL, a, src);
        const int32_t uL = __shfl_sync(FULL, uu, src);
        if (my < 0) aL = 0;
        uint32_t c = 0;
        for (int o0 = 0;; o0 += HUB_GLANES * HUB_UNROLL) {
            int32_t x[HUB_UNROLL];
#pragma unroll
            for (int j = 0; j < HUB_UNROLL; ++j) {
                const int o = o0 + j * HUB_GLANES + gl;
                x[j] = o < aL ? col[bL + o] : INT_MAX;
            }
#pragma unroll
            for (int j = 0; j < HUB_UNROLL; ++j) {
                if (x[j] <= maxv) {
                    const int p = probe(x[j]);
                    if (p >= 0) {
                        if (cnt) {
                            atomicAdd(&cnt[p], 1u);
                        } else {
                            atomicAdd(&t[x[j]], 1ull);
                            if (sup) atomicAdd(&sup[vbase + p], 1u);  // edge (v, x)
                        }
                        if (sup) atomicAdd(&sup[bL + o0 + j * HUB_GLANES + gl], 1u);  // edge (u, x)
                        ++c;
                    }
                }
            }
            // the suffix is sorted: a group is done once one of its lanes read past maxv
            // (or past the end of the suffix)
            if (__ballot_sync(FULL, x[HUB_UNROLL - 1] > maxv) & gmask) aL = 0;
            if (__all_sync(FULL, aL == 0)) break;
        }
#pragma unroll
        for (int off = HUB_GLANES / 2; off > 0; off >>= 1) c += __shfl_xor_sync(FULL, c, off);
        if (gl == 0 && my >= 0 && c) {
            atomicAdd(&t[uL], (unsigned long long)c);
            if (sup) atomicAdd(&sup[bL - 1], c);  // edge (u, v): bL is the entry after v
        }
        total_c += __reduce_add_sync(FULL, gl == 0 ? c : 0u);
    }
    if (a >= HUB_LONG) a = 0;  // done above
    const unsigned nz = __ballot_sync(FULL, a > 0);
    const int cz = __popc(nz);
    if (cz == 0) return total_c;
    // lane i takes the i-th short in-edge
    const int src = lane < cz ? (int)__fns(nz, 0, lane + 1) : lane;
    uu = __shfl_sync(FULL, uu, src);
    b0 = __shfl_sync(FULL, b0, src);
    a = __shfl_sync(FULL, a, src);
    if (lane >= cz) a = 0;
    int incl = warp_inclusive_scan(a);
    const int total = __shfl_sync(FULL, incl, 31);
    const int excl = incl - a;
    if (lane >= cz) incl = INT_MAX;
    cw[lane] = 0;
    __syncwarp();
    for (int r = 0; r < total; r += 32) {
        const int i0 = __popc(__ballot_sync(FULL, incl <= r));
        unsigned mk = (lane > i0 && lane < cz && excl - r < 32) ? (1u << (excl - r)) : 0u;
        mk = __reduce_or_sync(FULL, mk);
        const int idx = min(i0 + __popc(mk & (lane == 31 ? FULL : ((2u << lane) - 1u))), 31);
        const int bi = __shfl_sync(FULL, b0, idx);
        const int xi = __shfl_sync(FULL, excl, idx);
        const int item = r + lane;
        if (item < total) {
            const int32_t x = col[bi + (item - xi)];
            if (x <= maxv) {
                const int p = probe(x);
                if (p >= 0) {
                    if (cnt) {
                        atomicAdd(&cnt[p], 1u);
                    } else {
                        atomicAdd(&t[x], 1ull);
                        if (sup) atomicAdd(&sup[vbase + p], 1u);  // edge (v, x)
                    }
                    if (sup) atomicAdd(&sup[bi + (item - xi)], 1u);  // edge (u, x)
                    atomicAdd(&cw[idx], 1u);
                }
            }
        }
    }
    __syncwarp();
    const uint32_t cu = cw[lane];
    if (lane < cz && cu) {
        atomicAdd(&t[uu], (unsigned long long)cu);
        if (sup) atomicAdd(&sup[b0 - 1], cu);  // edge (u, v)
    }
    __syncwarp();
    return total_c + __reduce_add_sync(FULL, lane < cz ? cu : 0u);
}

constexpr int WINK_THREADS = 512;  // three resident blocks per SM: 64 KB of counters each
constexpr int WINK_WARPS = WINK_THREADS / 32;
constexpr int WINK_BLOCKS = 3;
constexpr uint32_t WIN_MARK = 0x80000000u;

__device__ __forceinline__ int shared_s32(uint32_t addr) {
    int v;
    asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// Probes of a lane's eight window offsets: s[j] < 0 iff offset j is an entry of the
// staged N+(v), whose counter has then been raised; returns how many are.
struct WinCounters {  // a block's counters, the entries of N+(v) marked in bit 31
    uint32_t addr;
    __device__ __forceinline__ uint32_t operator()(const uint32_t (&o)[8], int (&s)[8]) const {
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) s[j] = shared_s32(addr + o[j]);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            asm volatile("{ .reg .pred p; setp.lt.s32 p, %1, 0; @p red.shared.add.u32 [%0], 1; }" ::"r"(addr + o[j]),
                         "r"(s[j])
                         : "memory");
            c += (uint32_t)s[j] >> 31;
        }
        return c;
    }
};

// A block's marks, one bit per warp and rank; matches count in the block's counters of
// the highest ranks (MED_TOP), else directly in t.
struct WinMarks {
    uint32_t marks, cnt, first;  // shared addresses; offset of the first rank with a counter
    int shift;                   // 31 - the warp's bit
    unsigned long long* t;       // of the window's first rank
    __device__ __forceinline__ uint32_t operator()(const uint32_t (&o)[8], int (&s)[8]) const {
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            uint32_t m;
            asm volatile("ld.shared.u16 %0, [%1];" : "=r"(m) : "r"(marks + (o[j] >> 1)));
            s[j] = (int)(m << shift);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (s[j] < 0) {
                if (o[j] >= first)
                    asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(cnt + (o[j] - first)) : "memory");
                else
                    atomicAdd(&t[win_place(o[j] >> 2)], 1ull);
                ++c;
            }
        return c;
    }
};

// The same as a bitmap of one warp with the entries before each word, for counters per
// entry of N+(v) (per-edge support); the entry's bit is shifted into bit 31 of s[j].
struct WinBitmap {
    uint32_t bm, pre, cnt;
    __device__ __forceinline__ uint32_t operator()(const uint32_t (&o)[8], int (&s)[8]) const {
        uint32_t c = 0, i[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            i[j] = win_place(o[j] >> 2);
            s[j] = (int)__funnelshift_l(0u, (uint32_t)shared_s32(bm + ((i[j] >> 3) & ~3u)), ~i[j]);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (s[j] < 0) {
                uint32_t before;  // entries before the word, then those below the bit
                asm volatile("ld.shared.u8 %0, [%1];" : "=r"(before) : "r"(pre + (i[j] >> 5)));
                const uint32_t pos = before + __popc(s[j]) - 1;
                asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(cnt + 4 * pos) : "memory");
                ++c;
            }
        return c;
    }
};

// One batch of up to 32 in-edges (each lane's record; {0, 0}: none) of the hub whose
// entries of the window `probe` holds (LOW: window 2 or 3, else window 1).  An item is a vector: a round takes 32 of them, one per lane, each
// lane probing its eight entries.  The scan over the per-lane matches of two rounds (16
// bits each) gives, at the last vector of every in-edge, the matches up to it, so an
// in-edge's count is the difference of two of them.  Returns the batch total (all lanes).
//
// What bounds it: shared-memory wavefronts (79% of the peak in k_tc_hub on R-MAT scale
// 20), the random counter loads (2.9 wavefronts each) and the matches' atomics.  32-bit
// ids against a bitmap with prefix counts took 1.9 warp instructions per entry, this 0.9.
// Two rounds per scan: 0.73 instead of 0.75-0.80 ms.  Unconditional atomics, or atomics
// to a spare slot for the entries that do not match, took 0.83 and 0.77 ms.
template <bool SUP, bool LOW, class Probe>
__device__ __forceinline__ uint32_t win_batch(const uint2 rec, int win_no, bool hub_in_window,
                                              const int2* __restrict__ rowinfo, const uint2* __restrict__ winrow,
                                              const uint4* __restrict__ winlow,
                                              const uint4* __restrict__ win, const Probe& probe,
                                              unsigned long long* __restrict__ t, int2* at, uint32_t* cw,
                                              uint32_t* __restrict__ sup) {
    const int lane = lane_id();
    // the row's entries in the window (len of them, from vector first on), and how many
    // of them the suffix has
    uint32_t first = 0, len = 0, suffix = 0;
    if (rec.y) {
        if (!LOW) {
            const uint2 r = winrow[rec.x];
            first = r.x, len = r.y, suffix = rec.y;
        } else {
            const uint4 r = winlow[rec.x];
            suffix = rec.y - r.y;
            first = r.x, len = low_len(r, 2);
            if (win_no == 3) {
                suffix = suffix > len ? suffix - len : 0u;
                first += vectors_of(len);
                len = low_len(r, 3);
            }
            if (!suffix) len = 0;
        }
    }
    // a hub in the window: its suffixes begin inside a vector, whose entries before are
    // not above the hub and meet no mark of it; else the row's whole part of the window
    const uint32_t off = hub_in_window && suffix ? len - suffix : 0u;
    const int nv0 = suffix ? (int)vectors_of(len) - (int)(off >> 3) : 0;
    EdgeItems E;
    const int src = E.gather(nv0, cw);
    if (E.cz == 0) return 0;
    const uint32_t uu = __shfl_sync(FULL, rec.x, src);
    int32_t b0 = 0, cbase = 0;  // support: col index after v, and of the first vector's first entry
    if (SUP) {
        int32_t end = 0;
        if (rec.y) {
            const int2 ri = rowinfo[rec.x];
            end = ri.x + ri.y;
        }
        b0 = __shfl_sync(FULL, end - (int32_t)rec.y, src);
        cbase = __shfl_sync(FULL, end - (int32_t)(len - (off & ~7u)), src);
    }
    E.lay(__shfl_sync(FULL, nv0, src), (int)__shfl_sync(FULL, first + (off >> 3), src), at);
    constexpr uint32_t NONE2 = (LOW ? (uint32_t)HUB_WIN2 : WIN_NONE) * 0x10001u;
    uint32_t running = 0;
    for (int r = 0; r < E.total; r += 64) {
        const int item = r + lane;
        int idx[2];
        int2 e[2];
        uint4 q[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            idx[h] = 0;
            e[h] = make_int2(0, 0);
            q[h] = make_uint4(NONE2, NONE2, NONE2, NONE2);
            if (h == 0 || r + 32 < E.total) {
                idx[h] = E.edge_of(r + 32 * h);
                e[h] = at[idx[h]];
                if (item + 32 * h < E.total) q[h] = win[(uint32_t)(e[h].x + item + 32 * h)];
            }
        }
        uint32_t c = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h == 1 && r + 32 >= E.total) break;
            const uint32_t o[8] = {q[h].x & 0xffffu, q[h].x >> 16, q[h].y & 0xffffu, q[h].y >> 16,
                                   q[h].z & 0xffffu, q[h].z >> 16, q[h].w & 0xffffu, q[h].w >> 16};
            int s[8];
            const uint32_t ch = probe(o, s);
            c |= ch << (16 * h);
            if (SUP) {
                // edges (u, x): eight lanes take a vector's eight entries, which lie in one or
                // two sectors (k_tc_hub for 150 shuffled cliques of 300: each lane its own
                // entries one by one 1.61 ms, so 0.78)
                const int32_t cb = __shfl_sync(FULL, cbase, idx[h]), ex = __shfl_sync(FULL, E.excl, idx[h]);
                const uint32_t p0 = (uint32_t)cb + 8u * (uint32_t)(item + 32 * h - ex);
                uint32_t m = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) m |= (uint32_t)(s[j] < 0) << j;
                const unsigned any = __ballot_sync(FULL, m != 0);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    if (!(any >> (4 * k) & 0xfu)) continue;
                    const int from = 4 * k + (lane >> 3);
                    const uint32_t mk = __shfl_sync(FULL, m, from);
                    const uint32_t pk = __shfl_sync(FULL, p0, from);
                    if (mk >> (lane & 7) & 1u) atomicAdd(&sup[pk + (lane & 7)], 1u);
                }
            }
        }
        const uint32_t pc = warp_scan_u32(c);
        const uint32_t tot = __shfl_sync(FULL, pc, 31);
        if (e[0].y == item + 1) cw[idx[0]] = running + (pc & 0xffffu);  // an in-edge's last vector
        running += tot & 0xffffu;
        if (e[1].y == item + 33) cw[idx[1]] = running + (pc >> 16);
        running += tot >> 16;
    }
    __syncwarp();
    if (lane < E.cz) {
        const uint32_t c = cw[lane] - (lane ? cw[lane - 1] : 0u);
        if (c) {
            if (SUP)
                atomicAdd(&sup[b0 - 1], c);  // edge (u, v)
            else
                atomicAdd(&t[uu], (unsigned long long)c);
        }
    }
    __syncwarp();
    return running;
}

// Positions in col and in the in-edge records are below 2^31; a step or a lane past the last
// ones is not, so they are compared as 32 unsigned bits.
__host__ __device__ __forceinline__ constexpr bool before_end(uint32_t at, uint32_t end) { return at < end; }
static_assert(!before_end((uint32_t)INT_MAX - 1u + HUB_SLICE, (uint32_t)INT_MAX) &&
                  !before_end((uint32_t)INT_MAX + WINK_THREADS, (uint32_t)INT_MAX),
              "no position past the end wraps to one before it");
// The record at `at` of a task's in-edges, {0, 0} past their end.
__device__ __forceinline__ uint2 record_at(const uint2* __restrict__ in_rec, uint32_t at, uint32_t end) {
    return before_end(at, end) ? in_rec[at] : make_uint2(0, 0);
}

// In-edges a warp claims at a time: smaller batches when a slice has fewer than two
// full ones per warp, so that every warp gets some.
__device__ __forceinline__ int hub_batch_size(int64_t din, int warps) {
    return din >= 2 * warps * HUB_BATCH ? HUB_BATCH : max(8, (int)((din + 2 * warps - 1) / (2 * warps)));
}

struct HubShared {
    uint32_t cnt[HUB_WIN + 1];  // one counter per window rank and one that no hub marks
    int2 at[WINK_WARPS][32];
    uint32_t cw[WINK_WARPS][32];
    uint32_t vt[WINK_WARPS];
    unsigned q;
    unsigned bq;  // next batch of the current task
};

// Window tasks of the big hubs, one per block: N+(v)'s window entries mark their
// counters, the slice's suffixes are streamed against the marks, and the marks are
// taken away again, so a task costs O(|N+(v)|) beside its suffixes.  The counters keep
// counting t over the block's tasks and are flushed once (with per-edge support, which
// counts the entries of each N+(v) apart, after every task).  Thread 0 claims the next
// task while the current one is counted.
template <bool SUP>
__global__ void __launch_bounds__(WINK_THREADS, WINK_BLOCKS) k_tc_hub(
    int32_t T0w, const int2* __restrict__ rowinfo, const uint2* __restrict__ winrow, const int32_t* __restrict__ col,
    const uint4* __restrict__ win, const int4* __restrict__ win_task, const uint2* __restrict__ in_rec,
    unsigned long long* __restrict__ t, DevStats* stats, uint32_t* __restrict__ sup) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    HubShared& sh = *reinterpret_cast<HubShared*>(smem_raw);
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const unsigned ntask = stats->hub_tasks;
    unsigned next = blockIdx.x;
    if (next >= ntask) return;
    const WinCounters P{(uint32_t)__cvta_generic_to_shared(sh.cnt)};
    for (int i = threadIdx.x; i < HUB_WIN + 1; i += WINK_THREADS) sh.cnt[i] = 0;
    for (;;) {
        if (threadIdx.x == 0) {
            sh.q = next;
            sh.bq = 0;
        }
        __syncthreads();
        const unsigned q = sh.q;
        if (q >= ntask) break;
        if (threadIdx.x == 0) next = gridDim.x + atomicAdd(&stats->hub_next, 1u);
        const int4 task = win_task[q];
        const int32_t v = task.x;
        const uint32_t ne = (uint32_t)task.w & ((1u << TASK_BITS) - 1u), p1 = (uint32_t)task.z + ((uint32_t)task.w >> TASK_BITS);
        const uint32_t e1 = (uint32_t)task.y + ne;
        for (uint32_t p = (uint32_t)task.z + threadIdx.x; before_end(p, p1); p += WINK_THREADS)
            sh.cnt[win_place((uint32_t)(col[p] - T0w))] |= WIN_MARK;
        __syncthreads();
        uint32_t vtot = 0;
        const uint32_t bs = (uint32_t)hub_batch_size(ne, WINK_WARPS);
        for (;;) {
            unsigned k = 0;
            if (lane == 0) k = atomicAdd(&sh.bq, 1u);
            k = __shfl_sync(FULL, k, 0) * bs;
            if (k >= ne) break;
            const uint2 rec = (uint32_t)lane < bs ? record_at(in_rec, (uint32_t)task.y + k + lane, e1) : make_uint2(0, 0);
            vtot += win_batch<SUP, false>(rec, 1, v >= T0w, rowinfo, winrow, nullptr, win, P, t, sh.at[w], sh.cw[w], sup);
        }
        if (lane == 0) sh.vt[w] = vtot;
        __syncthreads();
        for (uint32_t p = (uint32_t)task.z + threadIdx.x; before_end(p, p1); p += WINK_THREADS) {
            const uint32_t x = win_place((uint32_t)(col[p] - T0w));
            const uint32_t c = sh.cnt[x] & ~WIN_MARK;
            sh.cnt[x] = SUP ? 0u : c;
            if (SUP && c) atomicAdd(&sup[p], c);  // edge (v, x)
        }
        if (!SUP && threadIdx.x == 0) {
            unsigned long long s = 0;
            for (int k = 0; k < WINK_WARPS; ++k) s += sh.vt[k];
            if (s) atomicAdd(&t[v], s);
        }
    }
    if (!SUP)
        for (int i = threadIdx.x; i < HUB_WIN; i += WINK_THREADS)
            if (const uint32_t c = sh.cnt[win_place((uint32_t)i)]) atomicAdd(&t[T0w + i], (unsigned long long)c);
}

// Ranks with a counter in k_tc_hub_med: the MED_TOP highest, or so (their places are
// permuted in groups of eight).  With 8 KB more a block the kernel has less L1 cache, and
// R-MAT scale 23 takes 358 instead of 319 us.  In a graph without other ranks (ALL) each has
// one: disjoint cliques of 200, 16,000 vertices, 480 -> 77 us.
constexpr int MED_TOP = 4096;
constexpr int MED_TOP0 = (HUB_WIN - MED_TOP) & ~7;  // the first of them in the window
template <bool SUP, bool ALL>
struct MedShared {
    uint32_t marks[(HUB_WIN + 1) / 2];  // two ranks per word
    uint32_t cnt[HUB_WIN + 1 - (ALL ? 0 : MED_TOP0)];
    int2 at[WINK_WARPS][32];
    uint32_t cw[WINK_WARPS][32];
};
template <bool ALL>
struct MedShared<true, ALL> {
    struct {
        uint32_t bm[(HUB_WIN + 1) / 32];
        uint32_t pre[(HUB_WIN + 1) / 128];  // one byte per word of bm
        uint32_t cnt[HUB_WARP_MAX];
    } win[WINK_WARPS];
    int2 at[WINK_WARPS][32];
    uint32_t cw[WINK_WARPS][32];
};
static_assert(WINK_WARPS == 16, "one mark bit per warp");
static_assert(HUB_WARP_MAX <= 256, "one-byte prefix counts");

// Window tasks of the other hubs, one per warp (taken from the back of the task list).
// Each warp owns one bit of the block's marks, so sixteen hubs share one table and a
// hub costs O(|N+(v)|) beside its suffixes.
template <bool SUP, bool ALL>
__global__ void __launch_bounds__(WINK_THREADS, WINK_BLOCKS) k_tc_hub_med(
    int32_t T0w, int32_t W, const int2* __restrict__ rowinfo, const uint2* __restrict__ winrow,
    const int32_t* __restrict__ col, const uint4* __restrict__ win, const int4* __restrict__ win_task, int64_t task_cap,
    const uint2* __restrict__ in_rec, unsigned long long* __restrict__ t, DevStats* stats, uint32_t* __restrict__ sup) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    MedShared<SUP, ALL>& sh = *reinterpret_cast<MedShared<SUP, ALL>*>(smem_raw);
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const unsigned nmed = stats->hub_med;
    if (blockIdx.x * WINK_WARPS >= nmed) return;
    // in a graph of communities with ranks below window 1 k_tc_hub_win2 takes these tasks
    if (!SUP && !ALL && hub_dense(stats)) return;
    constexpr int top0 = ALL ? 0 : MED_TOP0;
    const int top = ALL ? (W + 7) & ~7 : HUB_WIN + 1 - MED_TOP0;  // counters in use
    if constexpr (!SUP) {
        for (int i = threadIdx.x; i < (HUB_WIN + 1) / 2; i += WINK_THREADS) sh.marks[i] = 0;
        for (int i = threadIdx.x; i < top; i += WINK_THREADS) sh.cnt[i] = 0;
        __syncthreads();
    }
    unsigned q = blockIdx.x * WINK_WARPS + w;
    while (q < nmed) {
        unsigned nx = 0;
        if (lane == 0) nx = gridDim.x * WINK_WARPS + atomicAdd(&stats->hub_next2, 1u);
        const int4 task = win_task[task_cap - 1 - q];
        const int32_t v = task.x;
        const int dwin = (int)((uint32_t)task.w >> TASK_BITS);
        const uint32_t e0 = (uint32_t)task.y, e1 = e0 + ((uint32_t)task.w & ((1u << TASK_BITS) - 1u));
        uint32_t vtot = 0;
        if constexpr (!SUP) {
            const WinMarks P{(uint32_t)__cvta_generic_to_shared(sh.marks), (uint32_t)__cvta_generic_to_shared(sh.cnt),
                             4u * top0, 31 - w, t + T0w};
            for (int p = lane; p < dwin; p += 32) {
                const uint32_t x = win_place((uint32_t)(col[task.z + p] - T0w));
                atomicOr(&sh.marks[x >> 1], 1u << (w + 16 * (x & 1)));
            }
            __syncwarp();
            uint2 rec = record_at(in_rec, e0 + lane, e1);
            for (uint32_t bb = e0; before_end(bb, e1); bb += 32) {
                const uint2 cur = rec;  // the next batch's records are loaded ahead
                rec = record_at(in_rec, bb + 32 + lane, e1);
                vtot += win_batch<SUP, false>(cur, 1, v >= T0w, rowinfo, winrow, nullptr, win, P, t, sh.at[w], sh.cw[w], sup);
            }
            for (int p = lane; p < dwin; p += 32) {
                const uint32_t x = win_place((uint32_t)(col[task.z + p] - T0w));
                atomicAnd(&sh.marks[x >> 1], ~(1u << (w + 16 * (x & 1))));
            }
            __syncwarp();
            if (lane == 0 && vtot) atomicAdd(&t[v], (unsigned long long)vtot);
        } else {
            auto& M = sh.win[w];
            constexpr int WORDS = (HUB_WIN + 1) / 32, PER = WORDS / 32;
            static_assert(PER == 16, "four bytes a word, four words a lane");
            if (dwin > HUB_WARP_MAX) {  // the lists never make such a hub medium: do not overrun the counters
                if (lane == 0) atomicOr(&stats->err, ERR_OVERFLOW);
                q = __shfl_sync(FULL, nx, 0);
                continue;
            }
            for (int i = lane; i < WORDS; i += 32) M.bm[i] = 0;
            for (int i = lane; i < dwin; i += 32) M.cnt[i] = 0;
            __syncwarp();
            for (int p = lane; p < dwin; p += 32) {
                const int x = col[task.z + p] - T0w;
                atomicOr(&M.bm[x >> 5], 1u << (x & 31));
            }
            __syncwarp();
            // lane l counts the entries before words 16 l .. 16 l + 15
            uint32_t pc[PER], sum = 0;
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                pc[i] = sum;
                sum += __popc(M.bm[lane * PER + i]);
            }
            const uint32_t before = warp_scan_u32(sum) - sum;
#pragma unroll
            for (int i = 0; i < PER; i += 4)
                M.pre[lane * (PER / 4) + i / 4] = ((before + pc[i]) & 0xffu) | ((before + pc[i + 1]) & 0xffu) << 8 |
                                                  ((before + pc[i + 2]) & 0xffu) << 16 |
                                                  ((before + pc[i + 3]) & 0xffu) << 24;
            __syncwarp();
            const WinBitmap P{(uint32_t)__cvta_generic_to_shared(M.bm), (uint32_t)__cvta_generic_to_shared(M.pre),
                              (uint32_t)__cvta_generic_to_shared(M.cnt)};
            for (uint32_t bb = e0; before_end(bb, e1); bb += 32) {
                const uint2 rec = record_at(in_rec, bb + lane, e1);
                win_batch<SUP, false>(rec, 1, v >= T0w, rowinfo, winrow, nullptr, win, P, t, sh.at[w], sh.cw[w], sup);
            }
            for (int p = lane; p < dwin; p += 32) {
                const uint32_t c = M.cnt[p];
                if (c) atomicAdd(&sup[task.z + p], c);  // edge (v, x)
            }
            __syncwarp();
        }
        q = __shfl_sync(FULL, nx, 0);
    }
    if constexpr (!SUP) {
        __syncthreads();
        for (int i = threadIdx.x; i < top; i += WINK_THREADS)
            if (sh.cnt[i]) atomicAdd(&t[T0w + (int)win_place((uint32_t)(top0 + i))], (unsigned long long)sh.cnt[i]);
    }
}

// A warp's bitmap of N+(v)'s entries in a window of HUB_WIN2 ranks; matches count
// directly in t (below window 1 no rank is hot).
struct WinBits {
    uint32_t bm;
    unsigned long long* t;  // of the window's first rank
    __device__ __forceinline__ uint32_t operator()(const uint32_t (&o)[8], int (&s)[8]) const {
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j)
            s[j] = (int)__funnelshift_l(0u, (uint32_t)shared_s32(bm + ((o[j] >> 3) & ~3u)), ~o[j]);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (s[j] < 0) {
                atomicAdd(&t[o[j]], 1ull);
                ++c;
            }
        return c;
    }
};

// A warp's set of N+(v)'s entries in a window, with a counter each, for graphs in which most
// probes hit: a slot is (offset << 16) | matches, at most HUB_SLICE of them.
constexpr uint32_t SLOT_EMPTY = 0xffff0000u;  // no rank's offset
constexpr int WIN_SET_LG = 11;
constexpr int WIN_SET_MAX = 1024;             // entries: half of the slots
static_assert(HUB_SLICE <= 0xffff && HUB_WIN2 == 0xffff && 4 * HUB_WIN < 0xffff, "slot fields");
struct WinSet {
    uint32_t tab;  // shared address
    static __device__ __forceinline__ uint32_t home(uint32_t o) { return (o * 0x9e3779b1u) >> (32 - WIN_SET_LG); }
    static __device__ __forceinline__ uint32_t after(uint32_t h) { return (h + 1) & ((1u << WIN_SET_LG) - 1u); }
    __device__ __forceinline__ uint32_t operator()(const uint32_t (&o)[8], int (&s)[8]) const {
        uint32_t c = 0, w[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) w[j] = (uint32_t)shared_s32(tab + 4 * home(o[j]));
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            uint32_t h = home(o[j]);
            while (w[j] != SLOT_EMPTY && w[j] >> 16 != o[j]) {  // ends: half of the slots are empty
                h = after(h);
                w[j] = (uint32_t)shared_s32(tab + 4 * h);
            }
            s[j] = w[j] != SLOT_EMPTY ? -1 : 0;
            if (s[j] < 0) {
                asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(tab + 4 * h) : "memory");
                ++c;
            }
        }
        return c;
    }
    template <bool LOW>
    static __device__ __forceinline__ uint32_t offset(uint32_t i) { return LOW ? i : 4u * win_place(i); }
    // The entries p0 .. p1 - 1 of col, in window 1 or (LOW) below it.
    template <bool LOW>
    static __device__ __forceinline__ void insert(uint32_t* slots, const int32_t* __restrict__ col, int32_t first,
                                                  uint32_t p0, uint32_t p1) {
        for (uint32_t p = p0 + lane_id(); before_end(p, p1); p += 32) {
            const uint32_t o = offset<LOW>((uint32_t)(col[p] - first));
            uint32_t h = home(o);
            while (atomicCAS(&slots[h], SLOT_EMPTY, o << 16) != SLOT_EMPTY) h = after(h);  // entries are distinct
        }
        __syncwarp();
    }
    template <bool LOW>
    static __device__ __forceinline__ void flush(uint32_t* slots, const int32_t* __restrict__ col, int32_t first,
                                                 uint32_t p0, uint32_t p1, unsigned long long* __restrict__ t) {
        for (uint32_t p = p0 + lane_id(); before_end(p, p1); p += 32) {
            const uint32_t o = offset<LOW>((uint32_t)(col[p] - first));
            uint32_t h = home(o);
            while (slots[h] >> 16 != o) h = after(h);
            const uint32_t c = slots[h] & 0xffffu;
            if (c) atomicAdd(&t[col[p]], (unsigned long long)c);
        }
        __syncwarp();
        // Emptied from every entry's home slot on: whoever empties a slot goes on to the
        // next, so each run of taken slots is emptied to its end.
        for (uint32_t p = p0 + lane_id(); before_end(p, p1); p += 32)
            for (uint32_t h = home(offset<LOW>((uint32_t)(col[p] - first))); slots[h] != SLOT_EMPTY; h = after(h))
                slots[h] = SLOT_EMPTY;
        __syncwarp();
    }
};

// Below-window tasks: for each window k >= 2 that N+(v) reaches, a warp marks N+(v)'s
// entries there in a bitmap, streams the in-edges' entries of the window against it and
// clears the marks.  8 KB of shared memory a warp leave 24 warps per SM; four windows of
// half the size and 48 warps took longer (R-MAT scale 23: 1.38 instead of 1.18 ms), since
// hubs then read their in-edges once more per window.
//
// Matches against the bitmap add to t in global memory, one atomic each.  Below window 1 of
// an R-MAT graph they are few, but in a graph of communities (hub_dense) most probes match
// and the atomics bind, 150 G/s.  There the lists go into sets in the bitmaps' memory
// instead, and the medium hubs' window tasks are counted the same way (k_tc_hub_med leaves
// them).  Whole calls, one atomic per match / sets: disjoint cliques of 100 (100,000
// vertices) 1.75 / 0.92 ms, of 800 (32,000) 27.2 / 4.5; a ring lattice of 128 neighbours
// on either side (65,536) 4.50 / 1.5; R-MAT scale 20 and 23 within 0.3 %.
constexpr int WIN2_THREADS = 256;
constexpr int WIN2_WARPS = WIN2_THREADS / 32;
constexpr int WIN2_BLOCKS = 3;
static_assert(HUB_WIN2 == 0xffff, "the last offset of an 8 KB bitmap is no rank's");
static_assert((HUB_WIN2 + 1) / 32 == 1 << WIN_SET_LG && 2 * WIN_SET_MAX == 1 << WIN_SET_LG, "slots of a set");

struct Win2Shared {
    uint32_t bm[WIN2_WARPS][(HUB_WIN2 + 1) / 32];
    int2 at[WIN2_WARPS][32];
    uint32_t cw[WIN2_WARPS][32];
};

__global__ void __launch_bounds__(WIN2_THREADS) k_tc_hub_win2(
    Windows T, const int2* __restrict__ rowinfo, const uint2* __restrict__ winrow, const uint4* __restrict__ winlow,
    const int32_t* __restrict__ col, const uint4* __restrict__ win, const int4* __restrict__ win_task, int64_t task_cap,
    const int4* __restrict__ low_task, bool probe_mode, int big_in, const uint32_t* __restrict__ indeg, int32_t hub0,
    const uint2* __restrict__ in_rec, unsigned long long* __restrict__ t, DevStats* stats) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Win2Shared& sh = *reinterpret_cast<Win2Shared*>(smem_raw);
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const bool dense = hub_dense(stats);
    const unsigned nlow = stats->hub_low, nmed = dense ? stats->hub_med : 0;
    if (blockIdx.x * WIN2_WARPS >= max(nlow, nmed)) return;
    uint32_t* const bm = sh.bm[w];
    const uint32_t bm_addr = (uint32_t)__cvta_generic_to_shared(bm);
    const auto clear = [&](uint32_t word) {
        for (int i = lane; i < (HUB_WIN2 + 1) / 32; i += 32) bm[i] = word;
        __syncwarp();
    };
    clear(dense ? SLOT_EMPTY : 0u);  // empty sets or bitmaps
    // a task's in-edges in one window; the next batch's records are loaded ahead
    const auto stream = [&](auto low, const int4& task, uint32_t e1, int win_no, bool hub_in_window, const auto& probe) {
        uint32_t hits = 0;
        uint2 rec = record_at(in_rec, (uint32_t)task.y + lane, e1);
        for (uint32_t bb = (uint32_t)task.y; before_end(bb, e1); bb += 32) {
            const uint2 cur = rec;
            rec = record_at(in_rec, bb + 32 + lane, e1);
            hits += win_batch<false, decltype(low)::value>(cur, win_no, hub_in_window, rowinfo, winrow, winlow, win, probe,
                                                           t, sh.at[w], sh.cw[w], nullptr);
        }
        return hits;
    };
    unsigned q = blockIdx.x * WIN2_WARPS + w;
    while (q < nmed) {
        unsigned nx = 0;
        if (lane == 0) nx = gridDim.x * WIN2_WARPS + atomicAdd(&stats->hub_next2, 1u);
        const int4 task = win_task[task_cap - 1 - q];
        q = __shfl_sync(FULL, nx, 0);
        const int ne = task.w & ((1 << TASK_BITS) - 1), p1 = task.z + (int)((uint32_t)task.w >> TASK_BITS);
        if (p1 - task.z > WIN_SET_MAX) {  // the lists never make such a hub medium: do not overrun the set
            if (lane == 0) atomicOr(&stats->err, ERR_OVERFLOW);
            continue;
        }
        WinSet::insert<false>(bm, col, T.first[1], task.z, p1);
        const uint32_t hits = stream(std::false_type{}, task, (uint32_t)(task.y + ne), 1, task.x >= T.first[1], WinSet{bm_addr});
        WinSet::flush<false>(bm, col, T.first[1], task.z, p1, t);
        if (lane == 0 && hits) atomicAdd(&t[task.x], (unsigned long long)hits);
    }
    q = blockIdx.x * WIN2_WARPS + w;
    while (q < nlow) {
        unsigned nx = 0;
        if (lane == 0) nx = gridDim.x * WIN2_WARPS + atomicAdd(&stats->hub_next4, 1u);
        const int4 task = low_task[q];
        q = __shfl_sync(FULL, nx, 0);
        const int32_t v = task.x;
        const uint32_t e1 = (uint32_t)(task.y + task.z);
        const int2 rv = rowinfo[v];
        // in probe mode the list kernel counts the big hubs
        if (probe_mode && (indeg[v - hub0] >= (uint32_t)big_in || rv.y > HUB_WARP_MAX)) continue;
        uint32_t vtot = 0;
        int p1 = rv.x + task.w;  // end of N+(v)'s entries not yet taken
        for (int win_no = 2; win_no <= WINS && p1 > rv.x; ++win_no) {
            const int32_t first = win_no == 2 ? T.first[2] : T.first[3];
            int p0 = rv.x;
            if (v < first) p0 += lower_bound(col + rv.x, 0, p1 - rv.x, first);
            if (p0 == p1) continue;
            if (dense && p1 - p0 <= WIN_SET_MAX) {
                WinSet::insert<true>(bm, col, first, p0, p1);
                vtot += stream(std::true_type{}, task, e1, win_no, v >= first, WinSet{bm_addr});
                WinSet::flush<true>(bm, col, first, p0, p1, t);
                p1 = p0;
                continue;
            }
            if (dense) clear(0u);
            for (uint32_t p = p0 + lane; before_end(p, p1); p += 32) {
                const int x = col[p] - first;
                atomicOr(&bm[x >> 5], 1u << (x & 31));
            }
            __syncwarp();
            vtot += stream(std::true_type{}, task, e1, win_no, v >= first, WinBits{bm_addr, t + first});
            for (uint32_t p = p0 + lane; before_end(p, p1); p += 32) bm[(col[p] - first) >> 5] = 0;
            __syncwarp();
            if (dense) clear(SLOT_EMPTY);
            p1 = p0;
        }
        if (lane == 0 && vtot) atomicAdd(&t[v], (unsigned long long)vtot);
    }
}

// Below-window tasks of the per-edge support, which needs a counter per entry of N+(v):
// a warp puts the part of N+(v) below window 1 into a hash set and streams the
// in-edges' 32-bit entries below it end to end, 32 per round, one per lane (two rounds
// share one scan, as in win_batch).
constexpr int LOW_THREADS = 256;
constexpr int LOW_WARPS = LOW_THREADS / 32;
constexpr int LOW_BLOCKS = 5;

struct LowShared {
    int32_t keys[LOW_WARPS][HUB_HASH_MAX];
    uint32_t cnt[LOW_WARPS][HUB_HASH_MAX];
    int2 at[LOW_WARPS][32];
    uint32_t cw[LOW_WARPS][32];
};

__global__ void __launch_bounds__(LOW_THREADS) k_tc_hub_low(
    const int2* __restrict__ rowinfo, const uint2* __restrict__ winrow, const int32_t* __restrict__ col,
    const int4* __restrict__ low_task, int big_in, const uint32_t* __restrict__ indeg, int32_t hub0,
    const uint2* __restrict__ in_rec, DevStats* stats, uint32_t* __restrict__ sup) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LowShared& sh = *reinterpret_cast<LowShared*>(smem_raw);
    const int lane = lane_id(), w = threadIdx.x >> 5;
    int32_t* const K = sh.keys[w];
    uint32_t* const cnt = sh.cnt[w];
    int2* const at = sh.at[w];
    uint32_t* const cw = sh.cw[w];
    const unsigned nlow = stats->hub_low;
    if (blockIdx.x * LOW_WARPS >= nlow) return;
    for (int p = lane; p < HUB_HASH_MAX; p += 32) {  // every slot is empty again after each task
        K[p] = -1;
        cnt[p] = 0;
    }
    __syncwarp();
    unsigned q = blockIdx.x * LOW_WARPS + w;
    while (q < nlow) {
        unsigned nx = 0;
        if (lane == 0) nx = gridDim.x * LOW_WARPS + atomicAdd(&stats->hub_next4, 1u);
        nx = __shfl_sync(FULL, nx, 0);
        const int4 task = low_task[q];
        q = nx;
        const int64_t e0 = task.y, e1 = e0 + task.z;
        const int dlow = task.w;
        const int2 rv = rowinfo[task.x];
        if (dlow > HUB_LIST_MIN && (indeg[task.x - hub0] >= (uint32_t)big_in || rv.y > HUB_WARP_MAX))
            continue;  // the list kernel's
        int lg = 5;
        while ((1 << lg) < HUB_HASH_LOAD * dlow) ++lg;
        const unsigned shift = 32u - (unsigned)lg, mask = (1u << lg) - 1u;
        bool staged = false;  // the set is built when the first entry to probe turns up
        for (int64_t bb = e0; bb < e1; bb += 32) {
            const uint2 rec = bb + lane < e1 ? in_rec[bb + lane] : make_uint2(0, 0);
            int a = (int)rec.y;
            int32_t b0 = 0;
            if (a > 0) {
                a -= (int)winrow[rec.x].y;
                if (a > 0) {
                    const int2 ru = rowinfo[rec.x];
                    b0 = ru.x + ru.y - (int)rec.y;
                }
            }
            EdgeItems E;
            const int src = E.gather(a, cw);
            if (E.cz == 0) continue;
            if (!staged) {
                for (int p = lane; p < dlow; p += 32) {
                    const int32_t x = col[rv.x + p];
                    unsigned h = ((unsigned)x * 0x9e3779b1u) >> shift;
                    while (atomicCAS(&K[h], -1, x) != -1) h = (h + 1) & mask;  // keys are distinct
                }
                staged = true;
            }
            b0 = __shfl_sync(FULL, b0, src);
            E.lay(__shfl_sync(FULL, a, src), b0, at);
            const HashProbe H{K, shift, mask};
            uint32_t running = 0;
            for (int r = 0; r < E.total; r += 64) {
                const int item = r + lane;
                int idx[2];
                int2 e[2];
                int32_t x[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    idx[h] = 0;
                    e[h] = make_int2(0, 0);
                    x[h] = -2;
                    if (h == 0 || r + 32 < E.total) {
                        idx[h] = E.edge_of(r + 32 * h);
                        e[h] = at[idx[h]];
                        if (item + 32 * h < E.total) x[h] = col[e[h].x + item + 32 * h];
                    }
                }
                uint32_t c = 0;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int slot = x[h] >= 0 ? H(x[h]) : -1;
                    if (slot >= 0) {
                        atomicAdd(&cnt[slot], 1u);
                        atomicAdd(&sup[e[h].x + item + 32 * h], 1u);  // edge (u, x)
                        c += 1u << (16 * h);
                    }
                }
                const uint32_t pc = warp_scan_u32(c);
                const uint32_t tot = __shfl_sync(FULL, pc, 31);
                if (e[0].y == item + 1) cw[idx[0]] = running + (pc & 0xffffu);
                running += tot & 0xffffu;
                if (e[1].y == item + 33) cw[idx[1]] = running + (pc >> 16);
                running += tot >> 16;
            }
            __syncwarp();
            if (lane < E.cz) {
                const uint32_t c = cw[lane] - (lane ? cw[lane - 1] : 0u);
                if (c) atomicAdd(&sup[b0 - 1], c);  // edge (u, v)
            }
            __syncwarp();
        }
        if (staged) {
            for (int p = lane; p <= (int)mask; p += 32) {
                const int32_t x = K[p];
                if (x >= 0) {
                    const uint32_t c = cnt[p];
                    if (c) atomicAdd(&sup[rv.x + lower_bound(col + rv.x, 0, dlow, x)], c);  // edge (v, x)
                    K[p] = -1;
                    cnt[p] = 0;
                }
            }
            __syncwarp();
        }
    }
}

struct HubListShared {
    union {
        struct {
            uint32_t bm[HUB_BM_WORDS];
            uint16_t pre[HUB_BM_WORDS];
        } b;
        int32_t list[HUB_CNT_MAX];
    } s;
    uint32_t cnt[HUB_CNT_MAX];
    uint32_t slice[HUB_BM_WORDS / 32];
    uint32_t cw[HUB_WARPS][32];
    unsigned long long vt[HUB_WARPS];
    int q;
    unsigned bq;  // next batch of the current hub
};

// One block per hub.  Per-edge support (SUP): big hubs with more than HUB_LIST_MIN entries
// below the window, the suffixes' entries there against that part of N+(v), staged as a
// bitmap with prefix counts.  Else probe mode: every big hub, the whole suffixes against
// the sorted list N+(v).
template <bool SUP>
__global__ void __launch_bounds__(HUB_THREADS) k_tc_hub_list(
    int32_t n, int32_t hub_cap, const int2* __restrict__ rowinfo, const uint2* __restrict__ winrow,
    const int32_t* __restrict__ col, const int64_t* __restrict__ hub_start, const int32_t* __restrict__ list,
    const uint2* __restrict__ in_rec, unsigned long long* __restrict__ t, DevStats* stats, uint32_t* __restrict__ sup_arg) {
    uint32_t* const sup = SUP ? sup_arg : nullptr;
    constexpr bool probe_mode = !SUP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    HubListShared& sh = *reinterpret_cast<HubListShared*>(smem_raw);
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const unsigned nlist = probe_mode ? stats->hub_big : stats->hub_long;
    for (;;) {
        if (threadIdx.x == 0) {
            sh.q = (int)atomicAdd(&stats->hub_next3, 1u);
            sh.bq = 0;
        }
        __syncthreads();
        const int q = sh.q;
        if ((unsigned)q >= nlist) break;
        const int32_t v = list[q];
        const int hi = v - (n - hub_cap);
        const int64_t e0 = hub_start[hi], e1 = hub_start[hi + 1];
        const int2 ri = rowinfo[v];
        const int64_t base = ri.x;
        // a list below the window: rows with a hub have their window entries counted
        const int dv = probe_mode ? ri.y : ri.y - (int)winrow[v].y;
        const int32_t maxv = col[base + dv - 1];
        const bool staged = dv <= HUB_CNT_MAX;
        const int W = (maxv - v + 31) >> 5;  // maxv - v < hub_cap <= HUB_BM_BITS
        if (staged)
            for (int p = threadIdx.x; p < dv; p += HUB_THREADS) sh.cnt[p] = 0;
        if (!probe_mode) {
            build_bitmap<HUB_THREADS>(sh.s.b.bm, sh.s.b.pre, sh.slice, col + base, dv, v, W);
        } else {
            if (staged)
                for (int p = threadIdx.x; p < dv; p += HUB_THREADS) sh.s.list[p] = col[base + p];
            __syncthreads();
        }
        uint32_t* cnt = staged ? sh.cnt : nullptr;
        unsigned long long vtot = 0;
        const int bs = hub_batch_size(e1 - e0, HUB_WARPS);
        const BitmapProbe PB{sh.s.b.bm, sh.s.b.pre, v};
        const ListProbe PL{staged ? sh.s.list : col + base, dv};
        for (;;) {
            unsigned k = 0;
            if (lane == 0) k = atomicAdd(&sh.bq, 1u);
            const int64_t bb = e0 + (int64_t)__shfl_sync(FULL, k, 0) * bs;
            if (bb >= e1) break;
            const int64_t be = min(bb + bs, e1);
            if constexpr (SUP)
                vtot += hub_batch<true>(bb, be, in_rec, rowinfo, winrow, col, maxv, PB, cnt, t, sh.cw[w], sup, base);
            else
                vtot += hub_batch<false>(bb, be, in_rec, rowinfo, winrow, col, maxv, PL, cnt, t, sh.cw[w], sup, base);
        }
        if (lane == 0) sh.vt[w] = vtot;
        __syncthreads();
        if (staged) {
            for (int p = threadIdx.x; p < dv; p += HUB_THREADS) {
                const uint32_t c = sh.cnt[p];
                if (c) {
                    atomicAdd(&t[col[base + p]], (unsigned long long)c);
                    if (sup) atomicAdd(&sup[base + p], c);  // edge (v, x)
                }
            }
        }
        if (threadIdx.x == 0) {
            unsigned long long s = 0;
            for (int k = 0; k < HUB_WARPS; ++k) s += sh.vt[k];
            if (s) atomicAdd(&t[v], s);
        }
        __syncthreads();
    }
}

// ---- reductions ---------------------------------------------------------------

__global__ void k_sum_t(int32_t n, const unsigned long long* __restrict__ t, DevStats* stats) {
    unsigned long long s = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) s += t[i];
    s = warp_sum(s);
    if (lane_id() == 0 && s) atomicAdd(&stats->sum_t, s);
}

// Eq. 2 with the simple degree; both operands are exact integers below 2^53, so
// the IEEE round-to-nearest division gives the correctly rounded quotient.
__global__ void k_finalize(int32_t n, const int32_t* __restrict__ rank, const unsigned long long* __restrict__ t_rank,
                           const int32_t* __restrict__ deg, unsigned long long* __restrict__ t_out,
                           double* __restrict__ lcc_out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int32_t r = rank[v];
        const unsigned long long tv = t_rank[r];
        if (t_out) t_out[v] = tv;
        if (lcc_out) {
            const long long d = deg[r];
            // t = 0 gives +0.0 without a double division (FP64 runs at a small fraction of FP32)
            lcc_out[v] = d < 2 || tv == 0 ? 0.0 : __ddiv_rn((double)(2ull * tv), (double)(d * (d - 1)));
        }
    }
}

// Per-bucket work: edges and sum of d+(u) + d+(v) over them (one thread per u).
__global__ void k_plan_stats(int32_t n, const int64_t* __restrict__ rowstart, const int32_t* __restrict__ rowlen,
                             const int32_t* __restrict__ col, const DevStats* stats,
                             unsigned long long* __restrict__ out) {
    const int32_t R = n - (int32_t)stats->hub_count;
    unsigned long long e[TC_NUM_BUCKETS + 1] = {}, ids[TC_NUM_BUCKETS + 1] = {};
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += stride) {
        const int d = rowlen[u];
        for (int k = 0; k < d; ++k) {
            const int32_t v = col[rowstart[u] + k];
            const int b = v >= R ? TC_BUCKET_HUB
                                 : (d < 2 ? TC_NUM_BUCKETS : (d <= SMALL_WIDE_MAX ? TC_BUCKET_SMALL : TC_BUCKET_CTA));
            e[b] += 1;
            ids[b] += (unsigned long long)(d + rowlen[v]);
        }
    }
#pragma unroll
    for (int b = 0; b <= TC_NUM_BUCKETS; ++b) {
        const unsigned long long x = warp_sum(e[b]), y = warp_sum(ids[b]);
        if (lane_id() == 0) {
            if (x) atomicAdd(&out[b], x);
            if (y) atomicAdd(&out[TC_NUM_BUCKETS + 1 + b], y);
        }
    }
}

}  // namespace

void launch_plan_stats(const CountBuffers& C, unsigned long long* out, const Launch& L) {
    if (C.n <= 0) return;
    k_plan_stats<<<grid_for(C.n, THREADS, L.sms), THREADS, 0, L.stream>>>(C.n, C.rowstart, C.rowlen, C.col,
                                                                         C.stats, out);
    count_launch();
}

bool launch_plan(const CountBuffers& C, const Strategy& S, const Launch& L, const PlanStreams* ps) {
    if (C.n <= 0) return false;
    const int hub_max = S.hub_max < 0 ? 0 : S.hub_max;
    const bool hubs = C.hub_cap > 0 && hub_max > 0 && !C.no_hubs;
    const int core_max = hubs && C.core_cap > 0 && S.hub_core > 0 ? (S.hub_core < C.core_cap ? S.hub_core : C.core_cap) : 0;
    if (hubs) {  // else the hub count stays zero
        k_hub_count<<<grid_for(C.n, THREADS, L.sms), THREADS, 0, L.stream>>>(C.n, C.deg, S.hub_min_degree, C.hub_cap,
                                                                            hub_max, core_max, C.stats);
        count_launch();
    }
    // the hub lists and the dense core need only the hub count: with a second stream
    // they are built while the main stream lists and counts the push buckets
    const bool forked = hubs && ps != nullptr;
    Launch H = L;
    if (forked) {
        cudaEventRecord(ps->fork, L.stream);
        cudaStreamWaitEvent(ps->side, ps->fork, 0);
        H.stream = ps->side;
    }
    if (hubs) {
        if (core_max > 0) launch_core_plan(C, H);
        const Windows T(C.n);
        k_win_build<<<grid_for(C.n, WIN_THREADS, H.sms), WIN_THREADS, 0, H.stream>>>(
            C.n, T, C.rowinfo, C.col, C.winrow, C.winlow, C.win, C.win_cap, C.src_lo, C.src_hi, C.stats);
        count_launch();
        k_hub_indeg<<<grid_for(C.hub_cap, THREADS, H.sms), THREADS, 0, H.stream>>>(C.n, C.hub_cap, C.deg, C.rowlen,
                                                                                  C.core_cnt, C.hub_cnt, C.stats);
        count_launch();
        // and 64-bit cursors starting at every hub's first slot
        scan_u32_to_i64(C.hub_cnt, C.hub_start, C.hub_cap, C.tmp, H, reinterpret_cast<int64_t*>(C.hub_cur64));
        // Of a shard's plan only its sources' records are written, at the front of each hub's
        // segment; the list kernel of probe mode reads whole segments.
        const bool shard = C.src_lo > 0 || C.src_hi < C.n;
        if (shard && S.strat[TC_BUCKET_HUB] == TC_STRAT_PROBE)
            cudaMemsetAsync(C.in_rec, 0, sizeof(uint2) * (size_t)C.m_cap, H.stream);
        k_row_of<<<grid_for((int64_t)C.n, THREADS, H.sms), THREADS, 0, H.stream>>>(C.n, C.hub_cap, C.rowstart,
                                                                                  C.hub_start, C.rowof, C.src_lo,
                                                                                  C.src_hi, C.stats);
        count_launch();
        k_hub_scatter_rows<<<grid_for(C.n, THREADS, H.sms), THREADS, 0, H.stream>>>(
            C.n, C.hub_cap, C.rowstart, C.rowlen, C.col, C.hub_start, C.hub_cur64, C.in_rec, C.src_lo, C.src_hi,
            C.stats);
        count_launch();
        k_hub_scatter<<<grid_for((int64_t)C.m_cap / SCAT_ITEMS + 1, SCAT_THREADS, H.sms), SCAT_THREADS, 0, H.stream>>>(
            C.n, C.hub_cap, C.rowstart, C.rowinfo, C.col, C.rowof, C.hub_start, C.hub_cur64, C.in_rec, C.src_lo,
            C.src_hi, C.stats);
        count_launch();
        k_hub_lists<<<grid_for(C.hub_cap, THREADS, H.sms), THREADS, 0, H.stream>>>(
            C.n, C.hub_cap, T.first[1], C.rowinfo, C.col, C.winrow, C.hub_cnt, C.hub_start,
            S.hub_big_in > 0 ? S.hub_big_in : 1, C.big_list, C.long_list, C.win_task, C.low_task,
            hub_task_cap(C.hub_cap, C.m_cap), C.hub_cur64, shard, C.stats);
        count_launch();
    }
    if (forked) cudaEventRecord(ps->join, H.stream);
    const int samplers = hubs ? sample_blocks(C.n) : 0;
    k_plan<<<samplers + grid_for(C.n, THREADS * PLAN_ITEMS, L.sms), THREADS, 0, L.stream>>>(C.n, samplers, C.rowstart, C.rowlen, C.rowinfo, C.col,
                                                                   C.small_list[0], C.small_list[1],
                                                                   C.small_list[2], C.small_list[3], C.cta_list,
                                                                   C.src_lo, C.src_hi, C.stats);
    count_launch();
    return forked;
}

cudaError_t intersect_init_attributes() {
    const int wide = 2 * SMALL_WIDE_GROUPS * SMALL_WIDE_MAX * (int)sizeof(int32_t);
    cudaError_t e = cudaSuccess;
    if ((e = cudaFuncSetAttribute(k_tc_cta<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(CtaShared))) ||
        (e = cudaFuncSetAttribute(k_tc_cta<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(CtaShared))) ||
        (e = cudaFuncSetAttribute(k_tc_small_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, wide)) ||
        (e = cudaFuncSetAttribute(k_tc_hub<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(HubShared))) ||
        (e = cudaFuncSetAttribute(k_tc_hub<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(HubShared))) ||
        (e = cudaFuncSetAttribute(k_tc_hub_med<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(MedShared<false, false>))) ||
        (e = cudaFuncSetAttribute(k_tc_hub_med<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(MedShared<false, true>))) ||
        (e = cudaFuncSetAttribute(k_tc_hub_med<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(MedShared<true, false>))) ||
        (e = cudaFuncSetAttribute(k_tc_hub_win2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Win2Shared))) ||
        (e = cudaFuncSetAttribute(k_tc_hub_low, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LowShared))) ||
        (e = cudaFuncSetAttribute(k_tc_hub_list<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(HubListShared))))
        return e;
    return cudaFuncSetAttribute(k_tc_hub_list<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(HubListShared));
}

template <bool SUP>
void intersect_impl(const CountBuffers& C, const Strategy& S, cudaEvent_t* ev, const Launch& L) {
    if (C.n <= 0) return;
    if (ev) cudaEventRecord(ev[PH_SMALL], L.stream);
    const int ss = S.strat[TC_BUCKET_SMALL];
    const float sf = S.factor[TC_BUCKET_SMALL];
    const int64_t top = C.dplus_bound;  // classes of longer sources are empty: left out
    if (SUP || ss == TC_STRAT_HASH) {  // the support always hashes
        k_tc_small_sets<8, SUP><<<L.sms * SETS_BLOCKS, SMALL_WARPS * 32, 0, L.stream>>>(
            C.n, C.rowinfo, C.col, C.small_list[0], 0, C.t_rank, C.stats, C.sup);
        count_launch();
        if (top > 8) {
            k_tc_small_sets<16, SUP><<<L.sms * SETS_BLOCKS, SMALL_WARPS * 32, 0, L.stream>>>(
                C.n, C.rowinfo, C.col, C.small_list[1], 1, C.t_rank, C.stats, C.sup);
            count_launch();
        }
        if (top > 16) {
            k_tc_small_hash<HASH_LG_SHORT, SUP><<<L.sms * (SUP ? 4 : HASH_BLOCKS), SMALL_WARPS * 32, 0, L.stream>>>(
                C.n, C.rowinfo, C.col, C.small_list[2], 2, C.t_rank, C.stats, C.sup);
            count_launch();
        }
        if (top > 32) {
            k_tc_small_hash<HASH_LG_WIDE, SUP><<<L.sms * (SUP ? 4 : HASH_BLOCKS), SMALL_WARPS * 32, 0, L.stream>>>(
                C.n, C.rowinfo, C.col, C.small_list[3], 3, C.t_rank, C.stats, C.sup);
            count_launch();
        }
    } else {
        k_tc_small<8><<<L.sms * SMALL_BLOCKS, SMALL_WARPS * 32, 0, L.stream>>>(
            C.n, C.rowstart, C.rowlen, C.rowinfo, C.col, C.small_list[0], 0, C.t_rank, C.stats, ss, sf);
        count_launch();
        if (top > 8) {
            k_tc_small<16><<<L.sms * SMALL_BLOCKS, SMALL_WARPS * 32, 0, L.stream>>>(
                C.n, C.rowstart, C.rowlen, C.rowinfo, C.col, C.small_list[1], 1, C.t_rank, C.stats, ss, sf);
            count_launch();
        }
        if (top > 16) {
            k_tc_small<32><<<L.sms * SMALL_BLOCKS, SMALL_WARPS * 32, 0, L.stream>>>(
                C.n, C.rowstart, C.rowlen, C.rowinfo, C.col, C.small_list[2], 2, C.t_rank, C.stats, ss, sf);
            count_launch();
        }
        if (top > 32) {
            k_tc_small_wide<<<L.sms * SMALL_WIDE_BLOCKS, SMALL_WARPS * 32,
                              2 * SMALL_WIDE_GROUPS * SMALL_WIDE_MAX * sizeof(int32_t), L.stream>>>(
                C.n, C.rowinfo, C.col, C.small_list[3], C.t_rank, C.stats, ss, sf);
            count_launch();
        }
    }
    if (ev) cudaEventRecord(ev[PH_CTA], L.stream);
    if (top > SMALL_WIDE_MAX) {
        k_tc_cta<SUP><<<L.sms * 4, CTA_THREADS, sizeof(CtaShared), L.stream>>>(
            C.n, C.rowstart, C.rowlen, C.rowinfo, C.col, C.cta_list, C.t_rank, C.stats, S.strat[TC_BUCKET_CTA],
            S.factor[TC_BUCKET_CTA], C.sup);
        count_launch();
    }
    // the hub lists and the dense core come from the planner's second stream
    if (C.hub_ready) cudaStreamWaitEvent(L.stream, C.hub_ready, 0);
    if (ev) cudaEventRecord(ev[PH_HUB], L.stream);
    if (C.hub_cap > 0 && !C.no_hubs) {
        if (S.hub_core > 0) launch_core_count(C, L);
        const bool probe = S.strat[TC_BUCKET_HUB] == TC_STRAT_PROBE;
        const Windows T(C.n);
        const int64_t task_cap = hub_task_cap(C.hub_cap, C.m_cap);
        if (!probe) {
            k_tc_hub<SUP><<<L.sms * WINK_BLOCKS, WINK_THREADS, sizeof(HubShared), L.stream>>>(
                T.first[1], C.rowinfo, C.winrow, C.col, C.win, C.win_task, C.in_rec, C.t_rank, C.stats, C.sup);
            count_launch();
        }
        const bool all = !SUP && T.first[1] == 0;
        const auto med = all ? k_tc_hub_med<SUP, !SUP> : k_tc_hub_med<SUP, false>;
        med<<<L.sms * WINK_BLOCKS, WINK_THREADS, all ? sizeof(MedShared<SUP, !SUP>) : sizeof(MedShared<SUP, false>), L.stream>>>(
            T.first[1], C.n - T.first[1], C.rowinfo, C.winrow, C.col, C.win, C.win_task, task_cap, C.in_rec, C.t_rank, C.stats, C.sup);
        count_launch();
        if (T.first[1] > 0) {  // something lies below window 1
            if (SUP)
                k_tc_hub_low<<<L.sms * LOW_BLOCKS, LOW_THREADS, sizeof(LowShared), L.stream>>>(
                    C.rowinfo, C.winrow, C.col, C.low_task, S.hub_big_in > 0 ? S.hub_big_in : 1, C.hub_cnt,
                    C.n - C.hub_cap, C.in_rec, C.stats, C.sup);
            else
                k_tc_hub_win2<<<L.sms * WIN2_BLOCKS, WIN2_THREADS, sizeof(Win2Shared), L.stream>>>(
                    T, C.rowinfo, C.winrow, C.winlow, C.col, C.win, C.win_task, task_cap, C.low_task, probe, S.hub_big_in > 0 ? S.hub_big_in : 1,
                    C.hub_cnt, C.n - C.hub_cap, C.in_rec, C.t_rank, C.stats);
            count_launch();
        }
        if (SUP ? T.first[1] > 0 : probe) {
            k_tc_hub_list<SUP><<<L.sms * HUB_BLOCKS, HUB_THREADS, sizeof(HubListShared), L.stream>>>(
                C.n, C.hub_cap, C.rowinfo, C.winrow, C.col, C.hub_start, SUP ? C.long_list : C.big_list, C.in_rec,
                C.t_rank, C.stats, C.sup);
            count_launch();
        }
    }
    if (ev) cudaEventRecord(ev[PH_END], L.stream);
}

// The plain count, or the count that also records every triangle's three edges in
// C.sup (tc_edge_support), from the same kernels compiled twice.
void launch_intersect(const CountBuffers& C, const Strategy& S, cudaEvent_t* ev, const Launch& L) {
    if (C.sup)
        intersect_impl<true>(C, S, ev, L);
    else
        intersect_impl<false>(C, S, ev, L);
}

void launch_sum_t(const CountBuffers& C, const Launch& L) {
    if (C.n <= 0) return;
    k_sum_t<<<grid_for(C.n, THREADS, L.sms), THREADS, 0, L.stream>>>(C.n, C.t_rank, C.stats);
    count_launch();
}

void launch_finalize(int32_t n, const int32_t* rank, const unsigned long long* t_rank, const int32_t* deg,
                     unsigned long long* t_out, double* lcc_out, const Launch& L) {
    if (n <= 0) return;
    k_finalize<<<grid_for(n, THREADS, L.sms), THREADS, 0, L.stream>>>(n, rank, t_rank, deg, t_out, lcc_out);
    count_launch();
}

}  // namespace tcg

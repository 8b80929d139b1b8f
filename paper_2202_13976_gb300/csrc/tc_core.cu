// Dense core of the hub bucket: the core_n highest ranks (c0 = n - core_n .. n-1).
//
// Every out-neighbour of a core vertex has a higher rank, so it lies in the core too:
// a triangle whose lowest vertex is in the core lies wholly in the core.  On
// scale-free graphs the top ranks are densely linked, and their triangles make up a
// large part of the wedges the hub kernel would probe one by one (each in-edge
// (u -> v) reads the suffix of N+(u) after v, Sec. III / Eq. 1).  In the core the
// same counts come from bit-parallel intersections with the rows of one symmetric
// bit matrix over core indices i = rank - c0:
//   Z[i] : bit j set iff i and j are adjacent
// For a core edge (x -> y), x < y, let S(x, y) = |{w > x : x -> w, w adjacent to y}|,
// the popcount of (Z[x] above bit x) AND Z[y].  A triangle a < b < c of the core
// is seen in S(a, b) (w = c) and in S(a, c) (w = b) and in no other S, so
//   t[y] += S(x, y) for every core edge, and t[x] += (sum over y of S(x, y)) / 2
// gives every core triangle once at each of its vertices (b and c through their own
// edge from a, a through the two).  The hub in-edge lists then leave out the
// in-edges whose source lies in the core.
#include <climits>

#include "tc_device.cuh"
#include "tc_internal.h"

namespace tcg {
namespace {

constexpr int CORE_THREADS = 256;
constexpr int CORE_WARPS = CORE_THREADS / 32;
constexpr int CORE_LANE_WORDS = 8;  // bitmap words each lane holds: 32 * 8 * 32 bits = CORE_MAX
// A lane's words: four from word 4 lane and four from word 128 + 4 lane, so that a warp's
// 16-byte loads of a row are contiguous.
__device__ __forceinline__ int lane_word(int lane, int h) { return 4 * lane + (h & ~3) * 32 + (h & 3); }
static_assert(32 * CORE_LANE_WORDS * 32 == CORE_MAX, "lane words cover the core");

// Words of a row that are written and read: the core's bits, rounded up to a lane's.
__device__ __forceinline__ int core_row_words(int core_n) {
    return ((core_n + 31) / 32 + CORE_LANE_WORDS - 1) / CORE_LANE_WORDS * CORE_LANE_WORDS;
}

// Z is built in two passes without a global atomic.  One warp per core vertex i gathers
// N+(i) as bits in shared memory and writes the row's words from i's own word on.
// Setting both ends' bits, bounds and counts by global atomics took 140 us on R-MAT
// scale 20 (2.9 M core edges, bound by the atomics) beside 8 MB to clear; the two passes
// take 50 us.
__global__ void __launch_bounds__(CORE_THREADS) k_core_rows(int32_t n, const int2* __restrict__ rowinfo,
                                                            const int32_t* __restrict__ col, int words,
                                                            uint32_t* __restrict__ z, int32_t* __restrict__ hiout,
                                                            const DevStats* stats) {
    __shared__ uint32_t bits[CORE_WARPS][CORE_MAX / 32];
    const int core_n = (int)stats->core_n;
    const int32_t c0 = n - core_n;
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int used = core_row_words(core_n);
    uint32_t* const row = bits[w];
    for (int i = blockIdx.x * CORE_WARPS + w; i < core_n; i += gridDim.x * CORE_WARPS) {
        const int2 ri = rowinfo[c0 + i];
        const int first = i >> 5;  // every bit of N+(i) lies above i
        for (int k = first + lane; k < used; k += 32) row[k] = 0;
        __syncwarp();
        for (int p = lane; p < ri.y; p += 32) {
            const int j = col[ri.x + p] - c0;
            atomicOr(&row[j >> 5], 1u << (j & 31));
        }
        __syncwarp();
        for (int k = first + lane; k < used; k += 32) z[(int64_t)i * words + k] = row[k];
        if (lane == 0) hiout[i] = ri.y > 0 ? col[ri.x + ri.y - 1] - c0 : -1;
        __syncwarp();  // row is reused
    }
}

// The words below: one block per 32 rows.  A warp turns the 32 x 32 bits of word column a
// in the rows of an earlier block b (transposed by ballots) into word b of this block's
// rows.  From the mirrored words come the in-degree cnt and the lowest and highest
// neighbour of every row (lo: CORE_MAX less it, hi: one more; 0: none).
constexpr int MIRROR_PITCH = CORE_MAX / 32 + 1;  // words; odd, so that a column's writes meet different banks

constexpr int MIRROR_THREADS = 1024;
constexpr int MIRROR_WARPS = MIRROR_THREADS / 32;

__global__ void __launch_bounds__(MIRROR_THREADS) k_core_mirror(int words, uint32_t* __restrict__ z,
                                                              int32_t* __restrict__ lo, int32_t* __restrict__ hi,
                                                              const int32_t* __restrict__ hiout,
                                                              uint32_t* __restrict__ cnt, const DevStats* stats) {
    __shared__ uint32_t tile[32 * MIRROR_PITCH];
    const int core_n = (int)stats->core_n;
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int blocks = (core_n + 31) / 32;
    for (int q = blockIdx.x; q < blocks; q += gridDim.x) {
        const int a = blocks - 1 - q;  // the blocks with the most words first
        for (int b = w; b <= a; b += MIRROR_WARPS) {
            const int r = 32 * b + lane;  // of block b, whose rows all exist when b < a
            const uint32_t x = r < core_n ? z[(int64_t)r * words + a] : 0u;
            uint32_t y = 0;
#pragma unroll
            for (int k = 0; k < 32; ++k) {
                const uint32_t m = __ballot_sync(FULL, (x >> k) & 1u);
                if (lane == k) y = m;
            }
            tile[lane * MIRROR_PITCH + b] = b < a ? y : x | y;  // the diagonal keeps its upper bits
        }
        __syncthreads();
        for (int l = w; l < 32; l += MIRROR_WARPS) {
            const int i = 32 * a + l;
            if (i >= core_n) break;
            uint32_t c = 0;
            int low = INT_MAX, high = -1;  // neighbours below i, then above in the diagonal word
            for (int k = lane; k <= a; k += 32) {
                const uint32_t v = tile[l * MIRROR_PITCH + k];
                z[(int64_t)i * words + k] = v;
                c += __popc(k < a ? v : v & ((1u << l) - 1u));
                if (v) {
                    low = min(low, 32 * k + __ffs(v) - 1);
                    high = 32 * k + 31 - __clz(v);
                }
            }
            c = __reduce_add_sync(FULL, c);
            low = __reduce_min_sync(FULL, low);
            high = __reduce_max_sync(FULL, high);
            // a row with no neighbour up to its own word has its lowest in the words above
            if (low == INT_MAX && hiout[i] >= 0) {
                for (int k0 = a + 1; low == INT_MAX; k0 += 32) {  // ends: a bit is set at hiout[i]
                    const int k = k0 + lane;
                    const uint32_t v = k <= hiout[i] >> 5 ? z[(int64_t)i * words + k] : 0u;
                    low = __reduce_min_sync(FULL, v ? 32 * k + __ffs(v) - 1 : INT_MAX);
                    if (k0 > hiout[i] >> 5) break;
                }
            }
            if (lane == 0) {
                cnt[i] = c;
                lo[i] = low == INT_MAX ? 0 : CORE_MAX - low;
                hi[i] = max(high, hiout[i]) + 1;
            }
        }
        __syncthreads();  // the tile is reused
    }
}

// The lane's words of a row that fall in the word range [w0, w1], 0 for the others.
__device__ __forceinline__ void lane_words(const uint32_t* __restrict__ row, int lane, int w0, int w1,
                                           uint32_t (&v)[CORE_LANE_WORDS]) {
#pragma unroll
    for (int h = 0; h < CORE_LANE_WORDS; h += 4) {
        const int q = lane_word(lane, h);  // word index of this uint4
        uint4 x = make_uint4(0, 0, 0, 0);
        if (q + 3 >= w0 && q <= w1) x = *reinterpret_cast<const uint4*>(row + q);
        v[h] = x.x, v[h + 1] = x.y, v[h + 2] = x.z, v[h + 3] = x.w;
    }
}

// Sum of popc(a & b) over a lane's eight words: three carry-save adders leave the counts
// of four words (popc runs at a quarter of the logic operations' rate).
__device__ __forceinline__ uint32_t and_popc(const uint32_t (&a)[CORE_LANE_WORDS], const uint32_t (&b)[CORE_LANE_WORDS]) {
    static_assert(CORE_LANE_WORDS == 8, "adder tree");
    uint32_t x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = a[k] & b[k];
    const auto sum = [](uint32_t p, uint32_t q, uint32_t r) { return p ^ q ^ r; };
    const auto carry = [](uint32_t p, uint32_t q, uint32_t r) { return (p & q) | (p & r) | (q & r); };
    const uint32_t s0 = sum(x[0], x[1], x[2]), c0 = carry(x[0], x[1], x[2]);
    const uint32_t s1 = sum(x[3], x[4], x[5]), c1 = carry(x[3], x[4], x[5]);
    const uint32_t s2 = sum(s0, s1, x[6]), c2 = carry(s0, s1, x[6]);
    const uint32_t t0 = sum(c0, c1, c2), t1 = carry(c0, c1, c2);
    return __popc(s2) + __popc(x[7]) + 2 * __popc(t0) + 4 * __popc(t1);
}

constexpr int CORE_CHUNK = 8;  // entries of a row that a warp takes at a time
constexpr int CORE_AHEAD = 4;  // rows Z[y] in flight
// Small blocks, since most rows have few entries; seven per SM leave 72 registers.
constexpr int COUNT_THREADS = 128;
constexpr int COUNT_WARPS = COUNT_THREADS / 32;
constexpr int COUNT_BLOCKS = 7;

// One block per core vertex x; its warps take the entries y of N+(x) in turn.  A lane
// holds its words of Z[x] with the bits at or below x cleared (that is, N+(x)) in
// registers and reads the same words of Z[y] where the bit ranges can overlap:
// (x, hiout[x]] against [lo[y], hi[y]].  Words outside that range are zero in one
// operand, so skipping them changes no count.
//
// Per-edge support (SUP): the core edge (x -> y) lies in |Z[x] AND Z[y]| triangles of the
// core, a third core vertex on either side of x or y, so the whole row Z[x] is held and
// each edge is counted complete where it is met; no triangle has to be named.
//
// Bound by instruction issue: R-MAT scale 20 / 23 0.207 / 0.257 ms, a 600,011-pair graph
// 39 us.  One row at a time, eight popcounts a lane and one atomic per entry took 0.31 /
// 0.39 ms and 54 us; two rows in flight 0.209 / 0.262 ms, blocks of 256 0.231 / 0.285 ms.
// Rows whose range nowhere overlaps x's are passed over, four at a time: the support of a
// complete bipartite graph of 3,000 + 3,000 vertices took 0.79 ms, 0.35 so.
template <bool SUP>
__global__ void __launch_bounds__(COUNT_THREADS, COUNT_BLOCKS) k_core_count(
    int32_t n, const int64_t* __restrict__ rowstart, const int32_t* __restrict__ rowlen, const int32_t* __restrict__ col,
    int words, const uint32_t* __restrict__ z, const int32_t* __restrict__ lo, const int32_t* __restrict__ hi,
    const int32_t* __restrict__ hiout, unsigned long long* __restrict__ t, uint32_t* __restrict__ sup, int32_t src_lo,
    int32_t src_hi, const DevStats* stats) {
    __shared__ unsigned long long tx_w[COUNT_WARPS];
    const int core_n = (int)stats->core_n;
    const int32_t c0 = n - core_n;
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int used = core_row_words(core_n);
    for (int64_t i = blockIdx.x; i < core_n; i += gridDim.x) {
        const int32_t x = c0 + (int32_t)i;
        const int d = x >= src_lo && x < src_hi ? rowlen[x] : 0;  // sources outside the counted shard: none
        if (d < (SUP ? 1 : 2)) continue;  // no triangle has x lowest; uniform across the block
        const int64_t base = rowstart[x];
        uint32_t ox[CORE_LANE_WORDS];
        lane_words(z + i * words, lane, SUP ? 0 : (int)i >> 5, used - 1, ox);
#pragma unroll
        for (int h = 0; h < CORE_LANE_WORDS && !SUP; ++h) {  // keep the bits above x
            const int b0 = lane_word(lane, h) * 32;
            if (b0 + 31 <= (int)i)
                ox[h] = 0;
            else if (b0 <= (int)i)
                ox[h] &= (~0u << ((int)i - b0)) << 1;
        }
        const int xlo = SUP ? CORE_MAX - lo[i] : (int)i + 1, xhi = SUP ? hi[i] - 1 : hiout[i];
        unsigned long long tx = 0;
        for (int p0 = w * CORE_CHUNK; p0 < d; p0 += COUNT_WARPS * CORE_CHUNK) {
            const int mine = p0 + (lane & (CORE_CHUNK - 1));
            int j = 0, b0 = 1, b1 = 0;
            if (mine < d) {
                j = col[base + mine] - c0;
                b0 = max(xlo, CORE_MAX - lo[j]), b1 = min(xhi, hi[j] - 1);
            }
            const int w0 = b0 >> 5, w1 = b0 <= b1 ? min(b1 >> 5, used - 1) : -1;
            uint32_t sum = 0;  // lane k < CORE_CHUNK: the bits shared with entry p0 + k
            const unsigned live = __ballot_sync(FULL, w1 >= 0);
#pragma unroll
            for (int g = 0; g < CORE_CHUNK; g += CORE_AHEAD) {
                if (!(live >> g & ((1u << CORE_AHEAD) - 1u))) continue;  // ranges that nowhere overlap
                uint32_t v[CORE_AHEAD][CORE_LANE_WORDS];
#pragma unroll
                for (int k = 0; k < CORE_AHEAD; ++k)
                    lane_words(z + (int64_t)__shfl_sync(FULL, j, g + k) * words, lane, __shfl_sync(FULL, w0, g + k),
                               __shfl_sync(FULL, w1, g + k), v[k]);
#pragma unroll
                for (int k = 0; k < CORE_AHEAD; ++k) {
                    uint32_t s = and_popc(v[k], ox);
                    tx += s;
                    s = __reduce_add_sync(FULL, s);
                    if (lane == g + k) sum = s;
                }
            }
            if (lane < CORE_CHUNK && sum) {
                if (SUP)
                    atomicAdd(&sup[base + mine], sum);
                else
                    atomicAdd(&t[c0 + j], (unsigned long long)sum);
            }
        }
        if (SUP) continue;
        tx = warp_sum(tx);
        if (lane == 0) tx_w[w] = tx;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long s = 0;
            for (int k = 0; k < COUNT_WARPS; ++k) s += tx_w[k];
            if (s) atomicAdd(&t[x], s / 2);  // every triangle with x lowest was seen twice
        }
        __syncthreads();
    }
}

}  // namespace

int core_words_for(int32_t core_cap) {
    int w = (core_cap + 31) / 32;
    return (w + 7) & ~7;  // rows start on 32-byte boundaries; lanes read uint4
}

void launch_core_plan(const CountBuffers& C, const Launch& L) {
    if (C.core_cap <= 0) return;
    k_core_rows<<<grid_for((int64_t)C.core_cap * 32, CORE_THREADS, L.sms), CORE_THREADS, 0, L.stream>>>(
        C.n, C.rowinfo, C.col, C.core_words, C.core_z, C.core_hiout, C.stats);
    count_launch();
    k_core_mirror<<<grid_for((C.core_cap + 31) / 32, 1, L.sms), MIRROR_THREADS, 0, L.stream>>>(
        C.core_words, C.core_z, C.core_lo, C.core_hi, C.core_hiout, C.core_cnt, C.stats);
    count_launch();
}

void launch_core_count(const CountBuffers& C, const Launch& L) {
    if (C.core_cap <= 0) return;
    const auto kernel = C.sup ? k_core_count<true> : k_core_count<false>;
    kernel<<<C.core_cap, COUNT_THREADS, 0, L.stream>>>(C.n, C.rowstart, C.rowlen, C.col, C.core_words, C.core_z,
                                                       C.core_lo, C.core_hi, C.core_hiout, C.t_rank, C.sup, C.src_lo,
                                                       C.src_hi, C.stats);
    count_launch();
}

}  // namespace tcg

// Stable radix sort of (key, index) pairs, least significant digit first: what the ordered push and the choice of the
// hot keys order their rows with.  One launch per digit.
//
// A tile of consecutive pairs belongs to one block of 1,024 threads; there are at most SORT_MAX_TILES tiles (one per
// multiprocessor; larger inputs get larger tiles, walked in rounds of 2,048 pairs).  hist[pass][tile][digit] holds the
// digit counts that a pass starts from: those of the first pass come with the kernel that makes the keys, those of every
// later pass are added up by the scatter of the pass before it, which knows where each pair goes and what its next digit
// is.  A scatter block turns them into its own first output positions by reading the counts of all tiles (at most 148 rows
// of at most 2 KB, from L2), which costs less than the two to four launches of a separate prefix sum.  The digits of a sort
// are as narrow as its number of passes allows, since the work on counts grows with their number.
#pragma once

#include "nups_internal.cuh"

constexpr unsigned SORT_THREADS = 1024, SORT_ITEMS = 2, SORT_DIGIT_BITS = 9, SORT_DIGITS = 1u << SORT_DIGIT_BITS;
constexpr unsigned SORT_WARPS = SORT_THREADS / 32, SORT_ROUND = SORT_THREADS * SORT_ITEMS, SORT_MAX_TILES = 148;

struct SortPlan {
    unsigned passes, digit_bits, tiles, tile_shift;
    uint64_t n;
    size_t hist_words() const { return ((size_t)passes * tiles) << digit_bits; }
};

static inline SortPlan sort_plan(uint64_t n, int bits)
{
    SortPlan p;
    p.n = n;
    p.passes = ((unsigned)bits + SORT_DIGIT_BITS - 1) / SORT_DIGIT_BITS;
    if (p.passes < 1) p.passes = 1;
    p.digit_bits = ((unsigned)bits + p.passes - 1) / p.passes;
    if (p.digit_bits < 5) p.digit_bits = 5;                        // at most one group of threads per warp of the block
    p.tile_shift = 11;                                             // SORT_ROUND pairs
    while (n && ((n - 1) >> p.tile_shift) + 1 > SORT_MAX_TILES) ++p.tile_shift;
    p.tiles = n ? (unsigned)(((n - 1) >> p.tile_shift) + 1) : 1;
    return p;
}
static_assert(SORT_ROUND == 1u << 11, "a tile is a whole number of rounds");

// Makes the keys (source is called by whole warps for SORT_ITEMS positions at a time), counts the first pass's digits and
// clears the counts of the later passes and the word behind them, which is left to whoever uses the sorted pairs.  One
// block per tile.
template <class K, class Source>
__global__ void __launch_bounds__(SORT_THREADS)
sort_begin_kernel(Source source, K* __restrict__ keys, uint32_t* __restrict__ hist, SortPlan p)
{
    grid_dependency_wait();
    __shared__ uint32_t h[SORT_DIGITS];
    const unsigned digits = 1u << p.digit_bits;
    if (threadIdx.x < digits) h[threadIdx.x] = 0u;
    const size_t row = (size_t)p.tiles << p.digit_bits;
    for (size_t e = row + (size_t)blockIdx.x * SORT_THREADS + threadIdx.x; e < row * p.passes + 1; e += (size_t)gridDim.x * SORT_THREADS)
        hist[e] = 0u;
    __syncthreads();
    const uint64_t first = (uint64_t)blockIdx.x << p.tile_shift;
    const uint64_t last = min(first + (uint64_t(1) << p.tile_shift), p.n);
    const unsigned mask = digits - 1u;
    for (uint64_t b = first; b < last; b += SORT_ROUND) {
        K k[SORT_ITEMS];
        source(b + threadIdx.x, SORT_THREADS, last, k);
#pragma unroll
        for (int m = 0; m < (int)SORT_ITEMS; ++m) {
            const uint64_t i = b + threadIdx.x + (uint64_t)m * SORT_THREADS;
            if (i < last) {
                keys[i] = k[m];
                atomicAdd(&h[(unsigned)k[m] & mask], 1u);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < digits) hist[((size_t)blockIdx.x << p.digit_bits) + threadIdx.x] = h[threadIdx.x];
}

// One pass: every pair of the tile goes to its place by digit.  FIRST: a pair's index is its position.
template <class K, bool FIRST>
__global__ void __launch_bounds__(SORT_THREADS)
sort_scatter_kernel(const K* __restrict__ keys, const uint32_t* __restrict__ vals, K* __restrict__ keys_out,
                    uint32_t* __restrict__ vals_out, uint32_t* __restrict__ hist, SortPlan p, unsigned pass)
{
    grid_dependency_wait();
    __shared__ __align__(16) uint16_t wcnt[SORT_WARPS * SORT_DIGITS];  // [warp][digit] pairs of a digit in a warp's share of the round
    __shared__ uint32_t running[SORT_DIGITS];                          // next output position of every digit
    __shared__ uint32_t part[2][SORT_THREADS];
    __shared__ uint32_t wsum[SORT_DIGITS / 32];
    const unsigned tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned digits = 1u << p.digit_bits, shift = pass * p.digit_bits, mask = digits - 1u;
    const bool more = pass + 1 < p.passes;
    const uint32_t* cnt = hist + (((size_t)pass * p.tiles) << p.digit_bits);
    uint32_t* next = hist + (((size_t)(pass + 1) * p.tiles) << p.digit_bits);
    const uint64_t first = (uint64_t)blockIdx.x << p.tile_shift;
    const uint64_t last = min(first + (uint64_t(1) << p.tile_shift), p.n);
    K key[SORT_ITEMS];
    uint32_t val[SORT_ITEMS], rank[SORT_ITEMS];
    auto fetch = [&](uint64_t mine) {
#pragma unroll
        for (int k = 0; k < (int)SORT_ITEMS; ++k) {
            const uint64_t i = mine + 32 * k;
            key[k] = i < last ? keys[i] : K(0);
            val[k] = FIRST ? (uint32_t)i : (i < last ? vals[i] : 0u);
        }
    };
    fetch(first + (uint64_t)warp * 32 * SORT_ITEMS + lane);
    // groups of `digits` threads: thread `my` of a group looks after digit `my`, the groups share out the tiles (and the warps)
    const unsigned my = tid & mask, group = tid >> p.digit_bits, groups = SORT_THREADS >> p.digit_bits;
    {
        uint32_t all = 0, before = 0;                              // pairs of the digit in all tiles, and in those before this one
#pragma unroll 8
        for (unsigned t = group; t < p.tiles; t += groups) {
            const uint32_t x = __ldcg(cnt + ((size_t)t << p.digit_bits) + my);
            all += x;
            before += t < blockIdx.x ? x : 0u;
        }
        part[0][tid] = all;
        part[1][tid] = before;
        __syncthreads();
        uint32_t inc = 0;
        if (tid < SORT_DIGITS) {
            all = before = 0;
            if (tid < digits)
                for (unsigned g = 0; g < groups; ++g) { all += part[0][(g << p.digit_bits) + tid]; before += part[1][(g << p.digit_bits) + tid]; }
            inc = all;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                if (lane >= (unsigned)o) inc += y;
            }
            if (lane == 31) wsum[warp] = inc;
        }
        __syncthreads();
        if (tid < SORT_DIGITS) {
            uint32_t lower = lane < warp ? wsum[lane] : 0u;        // digits of the warps before this one
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) lower += __shfl_xor_sync(0xFFFFFFFFu, lower, o);
            running[tid] = inc - all + before + lower;
        }
    }
    for (uint64_t b = first; b < last; b += SORT_ROUND) {
        const uint64_t mine = b + (uint64_t)warp * 32 * SORT_ITEMS + lane;
        if (b != first) fetch(mine);
        uint4* z = reinterpret_cast<uint4*>(wcnt);
        for (unsigned e = tid; e < (SORT_WARPS * 2 / 16) << p.digit_bits; e += SORT_THREADS) z[e] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        uint16_t* my_cnt = wcnt + (warp << p.digit_bits);
#pragma unroll
        for (int k = 0; k < (int)SORT_ITEMS; ++k) {
            const bool in = mine + 32 * k < last;
            const unsigned d = (unsigned)(key[k] >> shift) & mask;
            // the lanes with the same digit, bit by bit (a warp-wide match instruction takes several times as long)
            unsigned m = __ballot_sync(0xFFFFFFFFu, in);
            if (!in) m = ~m;
#pragma unroll
            for (unsigned bit = 0; bit < SORT_DIGIT_BITS; ++bit) {
                if (bit >= p.digit_bits) break;
                const unsigned ones = __ballot_sync(0xFFFFFFFFu, (d >> bit) & 1u);
                m &= (d >> bit) & 1u ? ones : ~ones;
            }
            const int leader = __ffs(m) - 1;
            uint32_t old = 0;
            if (in && (int)lane == leader) {
                old = my_cnt[d];
                my_cnt[d] = (uint16_t)(old + __popc(m));
            }
            rank[k] = __shfl_sync(0xFFFFFFFFu, old, leader) + __popc(m & ((1u << lane) - 1u));
            __syncwarp();
        }
        __syncthreads();
        // a warp's counts -> pairs of the digit in the warps before it: each group of threads takes its share of the warps
        const unsigned w0 = group * (SORT_WARPS / groups), w1 = w0 + SORT_WARPS / groups;
        uint32_t sum = 0;
#pragma unroll 8
        for (unsigned w = w0; w < w1; ++w) sum += wcnt[(w << p.digit_bits) + my];
        part[0][tid] = sum;
        __syncthreads();
        uint32_t total = 0;
        {
            uint32_t at = 0;
            for (unsigned g = 0; g < groups; ++g) {
                const uint32_t x = part[0][(g << p.digit_bits) + my];
                at += g < group ? x : 0u;
                total += x;
            }
#pragma unroll 4
            for (unsigned w = w0; w < w1; ++w) {
                const uint32_t x = wcnt[(w << p.digit_bits) + my];
                wcnt[(w << p.digit_bits) + my] = (uint16_t)at;
                at += x;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < (int)SORT_ITEMS; ++k) {
            const bool in = mine + 32 * k < last;
            if (in) {
                const unsigned d = (unsigned)(key[k] >> shift) & mask;
                const uint32_t pos = running[d] + my_cnt[d] + rank[k];
                keys_out[pos] = key[k];
                vals_out[pos] = val[k];
                if (more)                                          // the next pass's counts
                    atomicAdd(next + ((size_t)(pos >> p.tile_shift) << p.digit_bits) + ((unsigned)(key[k] >> (shift + p.digit_bits)) & mask), 1u);
            }
        }
        __syncthreads();
        if (tid < digits) running[tid] += total;
    }
}

// The passes of a sort whose keys (and first counts) sort_begin_kernel has made in k0; k1, v0, v1 are work space.  The
// sorted pairs end up in (*k_out, *v_out): one of the two pairs of buffers.
template <class K>
static nups_status sort_passes(nups_store* s, K* k0, uint32_t* v0, K* k1, uint32_t* v1, uint32_t* hist, const SortPlan& p,
                               cudaStream_t st, K** k_out, uint32_t** v_out)
{
    for (unsigned pass = 0; pass < p.passes; ++pass) {
        if (pass == 0) nups_launch_dependent(sort_scatter_kernel<K, true>, p.tiles, SORT_THREADS, 0, st, k0, v0, k1, v1, hist, p, pass);
        else nups_launch_dependent(sort_scatter_kernel<K, false>, p.tiles, SORT_THREADS, 0, st, k0, v0, k1, v1, hist, p, pass);
        LAUNCH_CHECK(s);
        K* tk = k0; k0 = k1; k1 = tk;
        uint32_t* tv = v0; v0 = v1; v1 = tv;
    }
    *k_out = k0;
    *v_out = v0;
    return NUPS_OK;
}

// Device-wide building block used off the hot path (hot-set selection, per-key management,
// alias build): exclusive prefix sum over uint64.
#include "nups_internal.cuh"

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;   // 2048 values per block

__device__ __forceinline__ unsigned long long block_exclusive_scan(unsigned long long x, unsigned long long* total,
                                                                   unsigned long long* sh /* [33] */)
{
    // exclusive scan of one value per thread over a 256-thread block
    unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= (unsigned)o) inc += y;
    }
    if (lane == 31) sh[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        unsigned long long w = lane < (SCAN_THREADS / 32) ? sh[lane] : 0ull;
        unsigned long long winc = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, winc, o);
            if (lane >= (unsigned)o) winc += y;
        }
        if (lane < (SCAN_THREADS / 32)) sh[lane] = winc - w;
        if (lane == (SCAN_THREADS / 32) - 1) sh[32] = winc;
    }
    __syncthreads();
    unsigned long long res = sh[warp] + inc - x;
    *total = sh[32];
    __syncthreads();
    return res;
}

__global__ void scan_block_sums(const unsigned long long* __restrict__ in, unsigned long long* __restrict__ bsum,
                                uint64_t n)
{
    __shared__ unsigned long long sh[33];
    uint64_t base = (uint64_t)blockIdx.x * SCAN_TILE + (uint64_t)threadIdx.x * SCAN_ITEMS;
    unsigned long long t = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i)
        if (base + i < n) t += in[base + i];
    unsigned long long total;
    block_exclusive_scan(t, &total, sh);
    if (threadIdx.x == 0) bsum[blockIdx.x] = total;
}

// one block scans up to SCAN_TILE values in place
__global__ void scan_single_block(unsigned long long* data, uint64_t n, unsigned long long* total_out)
{
    __shared__ unsigned long long sh[33];
    uint64_t base = (uint64_t)threadIdx.x * SCAN_ITEMS;
    unsigned long long v[SCAN_ITEMS];
    unsigned long long t = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        v[i] = base + i < n ? data[base + i] : 0ull;
        t += v[i];
    }
    unsigned long long total;
    unsigned long long off = block_exclusive_scan(t, &total, sh);
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        if (base + i < n) data[base + i] = off;
        off += v[i];
    }
    if (threadIdx.x == 0 && total_out) *total_out = total;
}

__global__ void scan_apply(const unsigned long long* __restrict__ in, unsigned long long* __restrict__ out,
                           const unsigned long long* __restrict__ boff, uint64_t n)
{
    __shared__ unsigned long long sh[33];
    uint64_t base = (uint64_t)blockIdx.x * SCAN_TILE + (uint64_t)threadIdx.x * SCAN_ITEMS;
    unsigned long long v[SCAN_ITEMS];
    unsigned long long t = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        v[i] = base + i < n ? in[base + i] : 0ull;
        t += v[i];
    }
    unsigned long long total;
    unsigned long long off = block_exclusive_scan(t, &total, sh) + boff[blockIdx.x];
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        if (base + i < n) out[base + i] = off;
        off += v[i];
    }
}

}  // namespace

size_t nups_scan_scratch_bytes(uint64_t n)
{
    size_t bytes = 0;
    uint64_t m = n;
    while (m > (uint64_t)SCAN_TILE) {
        m = (m + SCAN_TILE - 1) / SCAN_TILE;
        bytes += ((m * 8 + 255) / 256) * 256;
    }
    return bytes + 256;
}

nups_status nups_scan_u64(nups_store* s, const unsigned long long* d_in, unsigned long long* d_out, uint64_t n,
                          unsigned long long* d_total, char* scratch, cudaStream_t st)
{
    if (n == 0) {
        if (d_total) CK(cudaMemsetAsync(d_total, 0, 8, st));
        return NUPS_OK;
    }
    if (n <= (uint64_t)SCAN_TILE) {
        if (d_out != d_in) CK(cudaMemcpyAsync(d_out, d_in, n * 8, cudaMemcpyDeviceToDevice, st));
        scan_single_block<<<1, SCAN_THREADS, 0, st>>>(d_out, n, d_total);
        LAUNCH_CHECK(s);
        return NUPS_OK;
    }
    uint64_t nb = (n + SCAN_TILE - 1) / SCAN_TILE;
    unsigned long long* bsum = (unsigned long long*)scratch;
    char* rest = scratch + ((nb * 8 + 255) / 256) * 256;
    scan_block_sums<<<(unsigned)nb, SCAN_THREADS, 0, st>>>(d_in, bsum, n);
    LAUNCH_CHECK(s);
    nups_status rc = nups_scan_u64(s, bsum, bsum, nb, d_total, rest, st);
    if (rc != NUPS_OK) return rc;
    scan_apply<<<(unsigned)nb, SCAN_THREADS, 0, st>>>(d_in, d_out, bsum, n);
    LAUNCH_CHECK(s);
    return NUPS_OK;
}

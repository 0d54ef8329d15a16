// Key store, direct access (pull / push), replica merge, access counting, hot-set selection and
// per-key management.  NuPS Sections 3.1, 3.2, 5.1.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <type_traits>

#include "nups_internal.cuh"
#include "nups_sort.cuh"

thread_local char g_nups_cuda_err[256] = "";

nups_status nups_cuda_fail(cudaError_t e, const char* what)
{
    snprintf(g_nups_cuda_err, sizeof(g_nups_cuda_err), "%s: %s", what, cudaGetErrorString(e));
    return NUPS_ECUDA;
}

extern "C" const char* nups_last_cuda_error(void) { return g_nups_cuda_err; }

extern "C" const char* nups_strerror(nups_status st)
{
    switch (st) {
        case NUPS_OK: return "ok";
        case NUPS_EINVAL: return "invalid argument";
        case NUPS_ENOMEM: return "out of memory or table full";
        case NUPS_ECUDA: return "CUDA runtime error";
        case NUPS_EKEY: return "key out of range seen on the device";
        case NUPS_ESTATE: return "call not valid in the current state";
        case NUPS_ETIMEOUT: return "bounded device-side wait gave up";
        default: return "unknown status";
    }
}

View nups_view(const nups_store* s)
{
    View v;
    v.val = s->val; v.acc = s->acc; v.dval = s->dval; v.dacc = s->dacc;
    v.hot_bits = s->hot_bits; v.slot_of = s->slot_of; v.dirty = s->dirty;
    v.cnt = s->cnt; v.own = s->own; v.epoch_tag = s->epoch << 8; v.st = s->st; v.loss_partial = s->loss_partial;
    v.num_keys = s->num_keys; v.Hcap = s->Hcap; v.H = (uint32_t)s->H; v.L4 = s->L / 4; v.R = s->R;
    v.count = s->cfg.count_accesses;
    v.merge_mean = s->cfg.merge_mean;
    v.f64 = s->vb == 8;
    v.clip_factor = s->cfg.clip_factor;
    return v;
}

nups_status nups_dev_alloc(nups_store* s, void** p, size_t bytes)
{
    *p = nullptr;
    if (bytes == 0) return NUPS_OK;
    if (s->dev_cap && (bytes > s->dev_cap || s->dev_bytes > s->dev_cap - bytes)) return NUPS_ENOMEM;   // the store's own limit
    if (cudaMalloc(p, bytes) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return NUPS_ENOMEM;
    }
    s->dev_bytes += bytes;
    return NUPS_OK;
}

void nups_dev_free(nups_store* s, void* p, size_t bytes)
{
    if (!p) return;
    cudaFree(p);                                   // waits for work that may still use it
    s->dev_bytes -= bytes < s->dev_bytes ? bytes : s->dev_bytes;
}

nups_status nups_scratch(nups_store* s, size_t bytes, char** out)
{
    if (bytes > s->scratch_bytes) {
        size_t want = bytes + bytes / 4 + (1u << 20);
        // the limit is judged with the old buffer already handed back; on refusal the old buffer stays
        auto refused = [&]() { return s->dev_cap && (want > s->dev_cap || s->dev_bytes - s->scratch_bytes > s->dev_cap - want); };
        // less to spare under a tight limit: the fixed parts of a choice among few hot keys take up to 15 KB more than sorting
        // all keys does, and are not to be what the limit refuses
        if (refused()) want -= 24u << 10;
        if (refused()) return NUPS_ENOMEM;
        nups_dev_free(s, s->scratch, s->scratch_bytes);
        s->scratch = nullptr; s->scratch_bytes = 0;
        nups_status rc = nups_dev_alloc(s, (void**)&s->scratch, want);
        if (rc != NUPS_OK) return rc;
        s->scratch_bytes = want;
    }
    *out = s->scratch;
    return NUPS_OK;
}

// Calls that move keys are numbered; the number is stored above the owner in every word such a call
// writes.  When the 24 bits run out, the numbers in the table are cleared and counting restarts.
__global__ void own_clear_epoch_kernel(uint32_t* own, uint64_t n)
{
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (; i < n; i += stride) own[i] &= 0xFFu;
}

nups_status nups_new_epoch(nups_store* s, cudaStream_t st)
{
    if (!s->own) return NUPS_OK;
    if (s->epoch >= 0xFFFFFFu) {
        own_clear_epoch_kernel<<<grid_for(s->num_keys, 256, 8192), 256, 0, st>>>(s->own, s->num_keys);
        LAUNCH_CHECK(s);
        s->epoch = 0;
    }
    s->epoch++;
    return NUPS_OK;
}

static inline size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// ---------------------------------------------------------------------------------------------
// optional event pairs around the main kernels (benchmark aid)
// ---------------------------------------------------------------------------------------------
static void timing_fold(nups_store* s)
{
    for (uint32_t i = 0; i < s->ev_n; ++i) {
        float ms = 0.f;
        const int kind = s->ev_kind[i];
        if (cudaEventSynchronize(s->ev[2 * i + 1]) == cudaSuccess &&
            cudaEventElapsedTime(&ms, s->ev[2 * i], s->ev[2 * i + 1]) == cudaSuccess)
            s->ev_ms[kind] += ms;
        s->ev_launches[kind]++;
    }
    s->ev_n = 0;
    cudaGetLastError();
}
void nups_time_begin(nups_store* s, cudaStream_t st, int kind)
{
    if (!s->timing) return;
    if (s->ev_n == NUPS_MAX_TIMED) timing_fold(s);
    s->ev_kind[s->ev_n] = (unsigned char)kind;
    cudaEventRecord(s->ev[2 * s->ev_n], st);
}
void nups_time_end(nups_store* s, cudaStream_t st)
{
    if (!s->timing) return;
    cudaEventRecord(s->ev[2 * s->ev_n + 1], st);
    s->ev_n++;
}
static void timing_clear(nups_store* s)
{
    for (int k = 0; k < NUPS_TIMED_KINDS; ++k) { s->ev_ms[k] = 0; s->ev_launches[k] = 0; }
}
extern "C" nups_status nups_kernel_timing(nups_store* s, int enable)
{
    if (!s) return NUPS_EINVAL;
    if (enable && !s->ev) {
        s->ev = (cudaEvent_t*)calloc(2 * NUPS_MAX_TIMED, sizeof(cudaEvent_t));
        s->ev_kind = (unsigned char*)calloc(NUPS_MAX_TIMED, 1);
        if (!s->ev || !s->ev_kind) return NUPS_ENOMEM;
        for (int i = 0; i < 2 * NUPS_MAX_TIMED; ++i) CK(cudaEventCreate(&s->ev[i]));
    }
    s->timing = enable ? 1 : 0;       // what was recorded stays until it is queried: switching costs no synchronisation
    return NUPS_OK;
}
extern "C" nups_status nups_kernel_times(nups_store* s, double* h_ms_out, uint64_t* h_launches_out, void* stream)
{
    if (!s || !h_ms_out || !h_launches_out) return NUPS_EINVAL;
    CK(cudaStreamSynchronize((cudaStream_t)stream));
    if (s->ev) timing_fold(s);
    for (int k = 0; k < NUPS_TIMED_KINDS; ++k) { h_ms_out[k] = s->ev_ms[k]; h_launches_out[k] = s->ev_launches[k]; }
    timing_clear(s);
    return NUPS_OK;
}
extern "C" nups_status nups_kernel_time(nups_store* s, double* h_ms_out, uint64_t* h_launches_out, void* stream)
{
    if (!s || !h_ms_out || !h_launches_out) return NUPS_EINVAL;
    double ms[NUPS_TIMED_KINDS];
    uint64_t n[NUPS_TIMED_KINDS];
    nups_status rc = nups_kernel_times(s, ms, n, stream);
    if (rc != NUPS_OK) return rc;
    *h_ms_out = 0; *h_launches_out = 0;
    for (int k = 0; k < NUPS_TIMED_KINDS; ++k) { *h_ms_out += ms[k]; *h_launches_out += n[k]; }
    return NUPS_OK;
}

// ---------------------------------------------------------------------------------------------
// create / destroy
// ---------------------------------------------------------------------------------------------
__global__ void fill_i32(int* p, uint64_t n, int value)
{
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (; i < n; i += stride) p[i] = value;
}

extern "C" nups_status nups_create(uint64_t num_keys, uint32_t value_len, const nups_config* cfg, nups_store** out)
{
    if (!out) return NUPS_EINVAL;
    *out = nullptr;
    if (num_keys == 0 || num_keys > 0xFFFFFFFFull || value_len == 0) return NUPS_EINVAL;
    nups_config c;
    memset(&c, 0, sizeof(c));
    if (cfg) c = *cfg;
    if (c.value_bytes == 0) c.value_bytes = 4;
    if (c.value_bytes != 4 && c.value_bytes != 8) return NUPS_EINVAL;
    if (((uint64_t)value_len * c.value_bytes) & 15) return NUPS_EINVAL;       // rows are multiples of 16 bytes
    if (c.value_bytes == 8 && (c.clip_factor > 0.f || c.sync_period_us)) return NUPS_EINVAL;
    if ((uint64_t)value_len * (c.value_bytes / 4) > 0xFFFFFFFFull) return NUPS_EINVAL;
    const uint32_t units = value_len * (c.value_bytes / 4);                     // row length in 4-byte units
    if (c.workers == 0) c.workers = 8;
    if (c.workers > 254) return NUPS_EINVAL;
    if (c.sync_period_us && c.deterministic) return NUPS_EINVAL;
    if (!(c.clip_factor >= 0.f)) return NUPS_EINVAL;
    if (c.merge_mean > 1 || (c.merge_mean && c.sync_period_us)) return NUPS_EINVAL;
    if (c.first_epoch > 0xFFFFFFu) return NUPS_EINVAL;
    // what the store holds from the start: tables, technique bitmap, slot map, counts, ownership words, status, loss words
    const size_t table_bytes = (size_t)num_keys * units * sizeof(float);
    const size_t bits_bytes = ((num_keys + 31) / 32) * 4, loss_bytes = 4 * NUPS_MAX_STEP_BLOCKS * sizeof(double);
    const size_t need = table_bytes * (c.with_adagrad ? 2 : 1) + bits_bytes + num_keys * 4 + num_keys * 8 +
                        (c.track_ownership ? num_keys * 4 : 0) + sizeof(DevStat) + loss_bytes;
    const size_t cap = (size_t)c.max_device_mib << 20;
    if (cap && need > cap) return NUPS_ENOMEM;              // the store's own limit, judged before the device is touched
    int dev = 0, count = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess || count == 0) {
        snprintf(g_nups_cuda_err, sizeof(g_nups_cuda_err), "no CUDA device");
        cudaGetLastError();
        return NUPS_ECUDA;
    }
    CK(cudaGetDevice(&dev));
    nups_store* s = (nups_store*)calloc(1, sizeof(nups_store));
    if (!s) return NUPS_ENOMEM;
    s->num_keys = num_keys; s->L = units; s->value_len = value_len; s->vb = c.value_bytes; s->R = c.workers; s->cfg = c;
    s->device = dev;
    s->dev_cap = cap;
    s->epoch = c.first_epoch;
    s->ahead_dist = -1;
    cudaDeviceGetAttribute(&s->sm_count, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&s->max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    bool ok = nups_dev_alloc(s, (void**)&s->val, table_bytes) == NUPS_OK;
    if (ok && c.with_adagrad) ok = nups_dev_alloc(s, (void**)&s->acc, table_bytes) == NUPS_OK;
    ok = ok && nups_dev_alloc(s, (void**)&s->hot_bits, bits_bytes) == NUPS_OK;
    ok = ok && nups_dev_alloc(s, (void**)&s->slot_of, num_keys * 4) == NUPS_OK;
    ok = ok && nups_dev_alloc(s, (void**)&s->cnt, num_keys * 8) == NUPS_OK;
    ok = ok && nups_dev_alloc(s, (void**)&s->st, sizeof(DevStat)) == NUPS_OK;
    ok = ok && nups_dev_alloc(s, (void**)&s->loss_partial, loss_bytes) == NUPS_OK;
    if (ok && c.track_ownership) ok = nups_dev_alloc(s, (void**)&s->own, num_keys * 4) == NUPS_OK;
    if (!ok) {
        cudaGetLastError();
        nups_destroy(s);
        return NUPS_ENOMEM;
    }
    cudaMemset(s->val, 0, table_bytes);
    if (s->acc) cudaMemset(s->acc, 0, table_bytes);
    cudaMemset(s->hot_bits, 0, ((num_keys + 31) / 32) * 4);
    cudaMemset(s->cnt, 0, num_keys * 8);
    cudaMemset(s->st, 0, sizeof(DevStat));
    cudaMemset(s->loss_partial, 0, 4 * NUPS_MAX_STEP_BLOCKS * sizeof(double));
    fill_i32<<<grid_for(num_keys, 256, 4096), 256>>>(s->slot_of, num_keys, -1);
    if (s->own) {
        fill_i32<<<grid_for(num_keys, 256, 4096), 256>>>((int*)s->own, num_keys, NUPS_OWNER_DEFAULT);
    }
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        nups_destroy(s);
        return nups_cuda_fail(e, "nups_create");
    }
    if (c.sync_period_us) {
        nups_status rc = nups_background_start(s, c.sync_period_us);
        if (rc != NUPS_OK) {
            nups_destroy(s);
            return rc;
        }
    }
    *out = s;
    return NUPS_OK;
}

extern "C" nups_status nups_destroy(nups_store* s)
{
    if (!s) return NUPS_OK;
    nups_background_stop(s);
    cudaDeviceSynchronize();
    if (s->side) { cudaStreamDestroy(s->side); cudaEventDestroy(s->side_fork); cudaEventDestroy(s->side_join); }
    for (int i = 0; i < NUPS_MAX_HANDLES; ++i) cudaFree(s->handle[i].buf);
    for (int i = 0; i < NUPS_MAX_DISTS; ++i) { cudaFree(s->dist[i].table); cudaFree(s->dist[i].off); }
    cudaFree(s->val); cudaFree(s->acc); cudaFree(s->hot_bits); cudaFree(s->slot_of); cudaFree(s->hot_keys);
    cudaFree(s->dval); cudaFree(s->dacc); cudaFree(s->dirty); cudaFree(s->cnt); cudaFree(s->own);
    cudaFree(s->st); cudaFree(s->loss_partial); cudaFree(s->scratch); cudaFree(s->negs_buf);
    cudaFree(s->merge_snap[0]); cudaFree(s->merge_snap[1]);
    if (s->ev) {
        for (int i = 0; i < 2 * NUPS_MAX_TIMED; ++i) cudaEventDestroy(s->ev[i]);
        free(s->ev);
        free(s->ev_kind);
    }
    cudaGetLastError();
    free(s);
    return NUPS_OK;
}

extern "C" nups_status nups_table_ptr(nups_store* s, int which, void** ptr, uint64_t* stride)
{
    if (!s || !ptr || (which != 0 && which != 1)) return NUPS_EINVAL;
    if (which == 1 && !s->acc) return NUPS_EINVAL;
    *ptr = which ? s->acc : s->val;
    if (stride) *stride = s->value_len;
    return NUPS_OK;
}

extern "C" nups_status nups_table_copy(nups_store* s, int which, void* d_buf, int to_store, void* stream)
{
    if (!s || !d_buf || (which != 0 && which != 1) || (which == 1 && !s->acc)) return NUPS_EINVAL;
    void* t = which ? s->acc : s->val;
    size_t bytes = (size_t)s->num_keys * s->L * sizeof(float);
    CK(cudaMemcpyAsync(to_store ? t : d_buf, to_store ? d_buf : t, bytes, cudaMemcpyDeviceToDevice,
                       (cudaStream_t)stream));
    return NUPS_OK;
}

__global__ void init_uniform_kernel(float4* t, uint64_t total4, uint64_t seed, uint32_t which, float unit)
{
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (; i < total4; i += stride) {
        uint32_t x[4];
        philox_at(seed, i, which, 3, 0, x);
        float4 r;
        r.x = __fmul_rn((float)((int)(x[0] >> 8) - 8388608), unit);
        r.y = __fmul_rn((float)((int)(x[1] >> 8) - 8388608), unit);
        r.z = __fmul_rn((float)((int)(x[2] >> 8) - 8388608), unit);
        r.w = __fmul_rn((float)((int)(x[3] >> 8) - 8388608), unit);
        t[i] = r;
    }
}

// the same values (each exactly representable in fp32) into a table of doubles
__global__ void init_uniform_f64_kernel(double* t, uint64_t total4, uint64_t seed, uint32_t which, float unit)
{
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (; i < total4; i += stride) {
        uint32_t x[4];
        philox_at(seed, i, which, 3, 0, x);
#pragma unroll
        for (int k = 0; k < 4; ++k) t[4 * i + k] = (double)__fmul_rn((float)((int)(x[k] >> 8) - 8388608), unit);
    }
}

extern "C" nups_status nups_init_uniform(nups_store* s, int which, uint64_t seed, float scale, void* stream)
{
    if (!s || (which != 0 && which != 1) || (which == 1 && !s->acc)) return NUPS_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const uint64_t values = s->num_keys * (uint64_t)s->value_len;
    if (values & 3) return NUPS_EINVAL;                       // the generator makes four values at a time
    const uint64_t total4 = values / 4;
    float unit = scale * (1.0f / 8388608.0f);
    const unsigned grid = grid_for(total4, 256, (unsigned)s->sm_count * 16);
    if (s->vb == 8)
        init_uniform_f64_kernel<<<grid, 256, 0, st>>>((double*)(which ? s->acc : s->val), total4, seed, (uint32_t)which, unit);
    else
        init_uniform_kernel<<<grid, 256, 0, st>>>((float4*)(which ? s->acc : s->val), total4, seed, (uint32_t)which, unit);
    LAUNCH_CHECK(s);
    return NUPS_OK;
}

// ---------------------------------------------------------------------------------------------
// pull: row gather.  One warp walks windows of 32 keys; each lane fetches one key of the window and
// turns it into the offset of its row (and of the worker's pending replica row, if the key is
// replicated); the warp then copies the rows four at a time with 128-bit loads and streaming
// stores.  TWO = also copy the matching rows of a second table.
// ---------------------------------------------------------------------------------------------
constexpr int GATHER_UNROLL = 4;
constexpr unsigned long long NO_ROW = ~0ull;

struct TablePair {
    const float4* table;   // stored rows
    const float4* slab;    // pending replica updates [R][Hcap][L]
    float4* out;           // [n][L]
};

template <bool HOT, bool TWO, bool F64, bool PARTS>
__global__ void __launch_bounds__(256, 4)
gather_kernel(View v, const uint32_t* __restrict__ keys, uint64_t n, TablePair A, TablePair B, int map,
              uint64_t map_base, uint64_t map_total, int do_count, uint32_t* __restrict__ keys_copy, uint32_t parts)
{
    grid_dependency_wait();
    const unsigned lane = threadIdx.x & 31;
    const uint64_t team = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, teams = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const uint64_t warp = PARTS ? team / parts : team, nwarps = PARTS ? teams / parts : teams;
    const uint32_t part = PARTS ? (uint32_t)(team - warp * parts) : 0u;            // this warp's share of the window's rows
    const uint32_t L4 = v.L4;
    // Lookups run ahead of the copies: while window w is copied, the key of window w + 2 and the
    // hot-bit word of window w + 1 are already on their way.
    const uint64_t stride = nwarps * 32;
    uint64_t base = warp * 32;
    uint32_t key_a = base + lane < n ? __ldg(keys + base + lane) : 0u;                         // window w
    uint32_t key_b = base + stride + lane < n ? __ldg(keys + base + stride + lane) : 0u;       // window w + 1
    uint32_t bits_a = (HOT && key_a < v.num_keys) ? __ldg(v.hot_bits + (key_a >> 5)) : 0u;
    for (; base < n; base += stride) {
        const uint64_t i = base + lane;
        const bool in = i < n;
        const uint32_t key = key_a;
        const uint32_t bits = bits_a;
        key_a = key_b;
        bits_a = (HOT && key_a < v.num_keys) ? __ldg(v.hot_bits + (key_a >> 5)) : 0u;
        key_b = base + 2 * stride + lane < n ? __ldg(keys + base + 2 * stride + lane) : 0u;
        const bool valid = in && key < v.num_keys;
        if (in && !valid && part == 0) flag_bad_key(v);
        if (keys_copy && in && part == 0) keys_copy[i] = key;                   // PullSample hands the keys out as well
        unsigned long long src = valid ? (unsigned long long)key * L4 : NO_ROW;   // NO_ROW: zero-filled output
        unsigned long long pend = NO_ROW;
        if (HOT && valid && ((bits >> (key & 31)) & 1u)) {
            const uint32_t slot = (uint32_t)__ldg(v.slot_of + key);
            const uint64_t idx = map_base + i;
            const uint32_t q = map == 0 ? worker_of_item(idx, map_total, v.R) : chunk_of_pos(idx, map_total, v.R);
            pend = ((unsigned long long)q * v.Hcap + slot) * L4;
        }
        if (do_count && v.count && part == 0) {
            if (valid) atomicAdd(v.cnt + key, 1ull);
            unsigned hot_m = __ballot_sync(0xFFFFFFFFu, valid && pend != NO_ROW);
            unsigned cold_m = __ballot_sync(0xFFFFFFFFu, valid && pend == NO_ROW);
            if (lane == 0) {
                if (hot_m) atomicAdd(&v.st->hot_hits, (unsigned long long)__popc(hot_m));
                if (cold_m) atomicAdd(&v.st->cold_hits, (unsigned long long)__popc(cold_m));
            }
        }
        const int rows = (int)min((uint64_t)32, n - base), share = PARTS ? 32 / (int)parts : 32;
        for (int r = (int)part * share; r < (PARTS ? min(rows, ((int)part + 1) * share) : rows); r += GATHER_UNROLL) {
            unsigned long long so[GATHER_UNROLL], po[GATHER_UNROLL];
#pragma unroll
            for (int u = 0; u < GATHER_UNROLL; ++u) {
                const int from = min(r + u, 31);
                so[u] = __shfl_sync(0xFFFFFFFFu, src, from);
                po[u] = HOT ? __shfl_sync(0xFFFFFFFFu, pend, from) : NO_ROW;
                if (r + u >= rows) so[u] = NO_ROW;
            }
            for (uint32_t c = lane; c < L4; c += 32) {
                float4 a[GATHER_UNROLL], b[GATHER_UNROLL];
#pragma unroll
                for (int u = 0; u < GATHER_UNROLL; ++u) {
                    a[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (TWO) b[u] = a[u];
                    if (so[u] != NO_ROW) {
                        // with a hot tier, rows of non-replicated keys are unlikely to be read again soon:
                        // fetch them with the streaming hint so that they do not push the technique
                        // bitmap and the replicated rows out of L2
                        if (HOT && po[u] == NO_ROW) a[u] = ld_stream_v4(A.table + so[u] + c);
                        else a[u] = __ldg(A.table + so[u] + c);
                        if (TWO) b[u] = __ldg(B.table + so[u] + c);
                        if (HOT && po[u] != NO_ROW) {
                            a[u] = add_chunk<F64>(a[u], A.slab[po[u] + c]);
                            if (TWO) b[u] = add_chunk<F64>(b[u], B.slab[po[u] + c]);
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < GATHER_UNROLL; ++u) {
                    if (r + u < rows) {
                        const uint64_t oo = (base + r + u) * L4 + c;
                        st_stream_v4(A.out + oo, a[u]);
                        if (TWO) st_stream_v4(B.out + oo, b[u]);
                    }
                }
            }
        }
    }
}

// The same gather with 256-bit loads and stores, for one table whose rows are a multiple of 32 bytes and at most 32
// such chunks long, with 32 a multiple of the chunk count (64, 128 or 256 floats): a warp instruction then moves
// 32 / C8 whole rows, which halves the load/store instructions per byte.  Used when some keys are replicated: once
// many rows come from L2 (hot or repeated keys) the copy is bound by the instructions its rows take in the
// load/store pipe, not by DRAM.
template <bool HOT, int C8, bool PARTS>
__global__ void __launch_bounds__(256, 4)
gather8_kernel(View v, const uint32_t* __restrict__ keys, uint64_t n, const float* __restrict__ table,
               const float* slab, float* __restrict__ out, int map, uint64_t map_base, uint64_t map_total, int do_count,
               uint32_t* __restrict__ keys_copy, uint32_t parts)
{
    grid_dependency_wait();
    constexpr int RPI = 32 / C8;                       // rows per warp instruction
    constexpr int UNR = 2;                             // instructions in flight
    const unsigned lane = threadIdx.x & 31;
    const unsigned sub = lane / C8, c = lane % C8;     // which of the instruction's rows, which chunk of it
    const uint64_t team = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, teams = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const uint64_t warp = PARTS ? team / parts : team, nwarps = PARTS ? teams / parts : teams;
    const uint32_t part = PARTS ? (uint32_t)(team - warp * parts) : 0u;            // this warp's share of the window's rows
    const uint64_t L = (uint64_t)v.L4 * 4;
    const uint64_t stride = nwarps * 32;
    uint64_t base = warp * 32;
    const uint64_t end = n;
    uint32_t key_a = base + lane < end ? __ldg(keys + base + lane) : 0u;
    uint32_t key_b = base + stride + lane < end ? __ldg(keys + base + stride + lane) : 0u;
    uint32_t bits_a = (HOT && key_a < v.num_keys) ? __ldg(v.hot_bits + (key_a >> 5)) : 0u;
    for (; base < end; base += stride) {
        const uint64_t i = base + lane;
        const bool in = i < end;
        const uint32_t key = key_a;
        const uint32_t bits = bits_a;
        key_a = key_b;
        bits_a = (HOT && key_a < v.num_keys) ? __ldg(v.hot_bits + (key_a >> 5)) : 0u;
        key_b = base + 2 * stride + lane < end ? __ldg(keys + base + 2 * stride + lane) : 0u;
        const bool valid = in && key < v.num_keys;
        if (in && !valid && part == 0) flag_bad_key(v);
        if (keys_copy && in && part == 0) keys_copy[i] = key;                   // PullSample hands the keys out as well
        // row numbers instead of offsets: one 32-bit shuffle each; 0xFFFFFFFF = no such row
        uint32_t src = valid ? key : 0xFFFFFFFFu;
        uint32_t pend = 0xFFFFFFFFu;                    // replica row (worker * Hcap + slot) of a replicated key
        if (HOT && valid && ((bits >> (key & 31)) & 1u)) {
            const uint32_t slot = (uint32_t)__ldg(v.slot_of + key);
            const uint64_t idx = map_base + i;
            const uint32_t q = map == 0 ? worker_of_item(idx, map_total, v.R) : chunk_of_pos(idx, map_total, v.R);
            pend = q * (uint32_t)v.Hcap + slot;
        }
        if (do_count && v.count && part == 0) {
            if (valid) atomicAdd(v.cnt + key, 1ull);
            unsigned hot_m = __ballot_sync(0xFFFFFFFFu, valid && pend != 0xFFFFFFFFu);
            unsigned cold_m = __ballot_sync(0xFFFFFFFFu, valid && pend == 0xFFFFFFFFu);
            if (lane == 0) {
                if (hot_m) atomicAdd(&v.st->hot_hits, (unsigned long long)__popc(hot_m));
                if (cold_m) atomicAdd(&v.st->cold_hits, (unsigned long long)__popc(cold_m));
            }
        }
        const int share = PARTS ? 32 / (int)parts : 32, rows = (int)min((uint64_t)((part + 1) * share), end - base);
        for (int r0 = (int)part * share; r0 < rows; r0 += UNR * RPI) {
            uint32_t so[UNR], po[UNR];
            F8 a[UNR];
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                const int row = r0 + u * RPI + (int)sub;
                so[u] = __shfl_sync(0xFFFFFFFFu, src, row & 31);
                po[u] = HOT ? __shfl_sync(0xFFFFFFFFu, pend, row & 31) : 0xFFFFFFFFu;
                if (row >= rows) so[u] = 0xFFFFFFFFu;
            }
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                a[u].a = make_float4(0.f, 0.f, 0.f, 0.f);
                a[u].b = a[u].a;
                if (so[u] != 0xFFFFFFFFu) {
                    const float* p = table + (uint64_t)so[u] * L + 8 * c;
                    // rows of non-replicated keys are unlikely to be read again soon: streaming hint
                    a[u] = (HOT && po[u] == 0xFFFFFFFFu) ? ld8_stream(p) : ld8_cached(p);
                    if (HOT && po[u] != 0xFFFFFFFFu) {
                        const F8 d = ld8_plain(slab + (uint64_t)po[u] * L + 8 * c);
                        a[u].a = add4(a[u].a, d.a);
                        a[u].b = add4(a[u].b, d.b);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                const int row = r0 + u * RPI + (int)sub;
                if (row < rows) st8_stream(out + (base + row) * L + 8 * c, a[u]);
            }
        }
    }
}

// Into how many warps (a power of two, at most `most`) the rows of a window of 32 are divided, so that up to `resident` warps
// have work.  A warp takes its rows a few at a time, one memory latency after the other, so the windows of a small call would
// leave most multiprocessors idle while a few warps wait eight times in a row; every warp of a window repeats its lookups.
// (The kernels of larger calls are built without the division, which took 0.5 % of a pull of 1M rows.)
// Measured: pulling 50,000 rows of 100 floats 13.7 -> 9.9 us, pushing 5,000 10.3 -> 6.8 us, a round of pull and push over two
// tables with 20,000 rows 43 -> 30 us.
static uint32_t window_parts(uint64_t rows, uint64_t resident, uint32_t most)
{
    uint32_t parts = 1;
    while (parts < most && (rows + 31) / 32 * (2 * parts) <= resident) parts *= 2;
    return parts;
}

nups_status nups_gather_internal(nups_store* s, const uint32_t* d_keys, uint64_t n, float* d_out_val,
                                 float* d_out_acc, int worker_map, uint64_t map_base, uint64_t map_total,
                                 int do_count, cudaStream_t st, uint32_t* d_keys_copy)
{
    if (n == 0 || (!d_out_val && !d_out_acc)) return NUPS_OK;
    View v = nups_view(s);
    TablePair V = {(const float4*)s->val, (const float4*)s->dval, (float4*)d_out_val};
    TablePair C = {(const float4*)s->acc, (const float4*)s->dacc, (float4*)d_out_acc};
    const bool two = d_out_val && d_out_acc;
    TablePair A = d_out_val ? V : C, B = C;
    // 4 resident blocks per SM, grid-stride.  Fewer rows than keep them all busy: several warps share a window of 32 rows.
    const uint32_t parts = window_parts(n, (uint64_t)s->sm_count * 4 * 8, 8);
    unsigned grid = grid_for(n * parts, 32 * 8, (unsigned)s->sm_count * 4);
    // one table, rows of 8, 16 or 32 chunks of 32 bytes, everything 32-byte aligned, some keys replicated: the
    // 256-bit variant.  (Measured on 1M-key pulls of 128-float rows: with a hot tier 152 vs 163 us at Zipf 1.0 and
    // 20-25 % faster when keys repeat as under sample reuse; without a hot tier, where every row comes from DRAM,
    // 187 vs 180 us, so those calls keep the 128-bit kernel.)
    const uint32_t c8 = s->L / 8;
    float* out1 = two ? nullptr : A.out ? (float*)A.out : nullptr;
    if (s->H && s->vb == 4 && !two && s->L % 8 == 0 && (c8 == 8 || c8 == 16 || c8 == 32) && ((uintptr_t)out1 & 31) == 0 &&
        (uint64_t)s->R * s->Hcap < 0xFFFFFFFFull) {
        const float* table = (const float*)A.table;
        const float* slab = (const float*)A.slab;
        nups_time_begin(s, st, worker_map == 1 ? NUPS_TIMED_SAMPLE_ROWS : NUPS_TIMED_PULL);
#define NUPS_G8(C8_)                                                                                                     \
        nups_launch_dependent(parts > 1 ? gather8_kernel<true, C8_, true> : gather8_kernel<true, C8_, false>, grid, 256, 0, st, v, d_keys, n, table, slab, out1, worker_map, map_base, map_total, \
                                                        do_count, d_keys_copy, parts)
        if (c8 == 8) NUPS_G8(8);
        else if (c8 == 16) NUPS_G8(16);
        else NUPS_G8(32);
#undef NUPS_G8
        nups_time_end(s, st);
        LAUNCH_CHECK(s);
        return NUPS_OK;
    }
    nups_time_begin(s, st, worker_map == 1 ? NUPS_TIMED_SAMPLE_ROWS : NUPS_TIMED_PULL);
#define NUPS_GATHER(HOT_, TWO_, F64_)                                                                                  \
    nups_launch_dependent(parts > 1 ? gather_kernel<HOT_, TWO_, F64_, true> : gather_kernel<HOT_, TWO_, F64_, false>, grid, 256, 0, st, v, d_keys, n, A, B, worker_map, map_base, map_total, do_count, \
                                                          d_keys_copy, parts)
    if (s->vb == 8) {                        // only replica reads add; rows without a replica are copied whatever they hold
        if (s->H) { if (two) NUPS_GATHER(true, true, true); else NUPS_GATHER(true, false, true); }
        else { if (two) NUPS_GATHER(false, true, false); else NUPS_GATHER(false, false, false); }
    } else if (s->H) {
        if (two) NUPS_GATHER(true, true, false); else NUPS_GATHER(true, false, false);
    } else {
        if (two) NUPS_GATHER(false, true, false); else NUPS_GATHER(false, false, false);
    }
#undef NUPS_GATHER
    nups_time_end(s, st);
    LAUNCH_CHECK(s);
    return NUPS_OK;
}

extern "C" nups_status nups_pull2(nups_store* s, const uint32_t* d_keys, uint64_t n, void* d_out_val_, void* d_out_acc_,
                                  void* stream)
{
    float* d_out_val = (float*)d_out_val_;
    float* d_out_acc = (float*)d_out_acc_;
    if (!s || (n && !d_keys) || n >= (1ull << 32)) return NUPS_EINVAL;
    if (d_out_acc && !s->acc) return NUPS_EINVAL;
    if (n && !d_out_val && !d_out_acc) return NUPS_EINVAL;
    return nups_gather_internal(s, d_keys, n, d_out_val, d_out_acc, 0, 0, n, 1, (cudaStream_t)stream, nullptr);
}

extern "C" nups_status nups_pull(nups_store* s, const uint32_t* d_keys, uint64_t n, void* d_out, void* stream)
{
    if (n && !d_out) return NUPS_EINVAL;
    return nups_pull2(s, d_keys, n, d_out, nullptr, stream);
}

// ---------------------------------------------------------------------------------------------
// push, fast mode: 128-bit reductions straight to the destination row.  Within a window of 32
// rows, rows with the same destination are summed in registers first (__match_any_sync) so that
// a hot destination receives one reduction per window instead of one per row.
// TWO = a second table gets its own deltas from the same call.
// ---------------------------------------------------------------------------------------------
// Two rows in flight per warp and four resident blocks of 256 threads per multiprocessor (64 registers a thread): measured
// against four rows and three blocks (80 registers), the extra warps are worth more than the deeper unrolling at every skew
// (1M keys x 128 floats: 275 vs 279 us at s = 0, 195 vs 199 us at s = 1.0 with 1,000 replicated keys, 138 vs 152 us at s = 1.4).
constexpr int PUSH_UNROLL = 2;
// 8-byte values: elements of two rows that a lane has in flight per table.  A small call is bound by the latency of these loads:
// 20,000 rows of 100 values 16.8 us with two, 14.1 with four; 300,000 rows of 128 values 153.6 and 151.0 us, 50,021 rows pushed to two
// tables after a pull 101.6 and 92.4.  Two cover both rows where they have at most PUSH_SHORT values: 300,000 rows of 32 values take
// 44.0 us with four, 41.3 with two.  Where warps share a window, a second form for short rows costs the longer ones more than it gives
// (two tables: 50.7 -> 54.6 us for 20,000 rows of 100; 20,000 rows of 32 8.6 -> 7.8).  The two rows' offsets are worked out before the
// loads: per element they took registers that had to be spilled (300,000 rows of 128 values, 500 keys replicated, 137.8 -> 134).
constexpr int PUSH_WIDE = 4;
constexpr uint32_t PUSH_SHORT = 32;
constexpr int PUSH_THREADS = 256;
constexpr int PUSH_BLOCKS = 4;            // one table; calls that update two tables at once keep three (80 registers)

struct PushPair {
    const float4* delta;   // [n][L] updates
    float* table;          // stored rows
    float* slab;           // replica slabs
};

// What a lane takes of a row at a time: 16 bytes of 4-byte values, one reduction for all four; single 8-byte values, for which
// there is no wider reduction, so that the lanes of one reduction touch consecutive values (two per lane, 16 bytes apart from
// lane to lane, use half of every sector: 300,000 rows of 128 values 180 -> 135 us).
template <bool F64>
struct PushElement {
    using T = float4;
    static __device__ __forceinline__ T zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
    static __device__ __forceinline__ T load(const float4* p, uint64_t i) { return ld_stream_v4(p + i); }
    static __device__ __forceinline__ T add(T a, T b) { return add4(a, b); }
    static __device__ __forceinline__ void reduce(float* base, uint64_t i, T x) { red_add_v4(base + 4 * i, x); }
};
template <>
struct PushElement<true> {
    using T = double;
    static __device__ __forceinline__ T zero() { return 0.0; }
    static __device__ __forceinline__ T load(const float4* p, uint64_t i) { return __ldcs(reinterpret_cast<const double*>(p) + i); }
    static __device__ __forceinline__ T add(T a, T b) { return a + b; }
    static __device__ __forceinline__ void reduce(float* base, uint64_t i, T x)
    {
        asm volatile("red.global.add.f64 [%0], %1;" ::"l"(reinterpret_cast<double*>(base) + i), "d"(x) : "memory");
    }
};

// TIER = the block keeps shared-memory accumulators for the hottest replica slots (slot < tier_rows)
// of ONE worker (block b serves worker b mod R and visits only that worker's share of the windows);
// updates to those slots are added in shared memory and reach the worker's replica once, when the
// block ends.  This is what keeps thousands of additions to one hot row from queueing at one L2
// address.
// TIER = 2: nothing is replicated, so there are no slots to key the accumulators on; the block then uses them as a
// direct-mapped cache of rows: accumulator (key mod tier_rows) is claimed by the first key that asks for it and
// takes that key's updates until the block ends (other keys that map there go straight to their rows).  Frequent
// keys show up early and often, so they take most accumulators, and a skewed batch stops queueing at a few L2
// addresses even when its frequent keys were never marked for replication.
// PARTS = several warps share a window of rows (see window_parts).  Calls that do not divide their windows do without its
// registers: 400,000 rows of 128 floats pulled and pushed to two tables, no key replicated, 292 us with it (it spills) and 287
// without; 300,000 rows of 128 8-byte values pushed 151.2 and 150.3 us (neither spills).
template <bool HOT, bool TWO, int TIER, bool F64, bool PARTS>
__global__ void __launch_bounds__(PUSH_THREADS, TWO ? PUSH_BLOCKS - 1 : PUSH_BLOCKS)
push_atomic_kernel(View v, const uint32_t* __restrict__ keys, uint64_t n, PushPair A, PushPair B, uint64_t n_items,
                   uint32_t rows_per_item, uint32_t tier_rows, uint32_t parts)
{
    grid_dependency_wait();
    extern __shared__ __align__(16) float tier_mem[];                  // TIER: [tier_rows][L] sums, then touched bits
    const unsigned lane = threadIdx.x & 31;
    using E = PushElement<F64>;
    const uint32_t L4 = v.L4, LE = F64 ? 2 * L4 : L4;                  // a row's length in 16-byte chunks and in elements
    const uint32_t R = v.R;
    unsigned* touched = reinterpret_cast<unsigned*>(tier_mem + (size_t)tier_rows * L4 * 4);
    unsigned* tags = touched + (tier_rows + 31) / 32;                  // TIER == 2: key that owns each accumulator
    if (TIER) {
        float4* z = reinterpret_cast<float4*>(tier_mem);
        for (uint32_t e = threadIdx.x; e < tier_rows * L4; e += blockDim.x) z[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (uint32_t e = threadIdx.x; e < (tier_rows + 31) / 32; e += blockDim.x) touched[e] = 0u;
        if (TIER == 2)
            for (uint32_t e = threadIdx.x; e < tier_rows; e += blockDim.x) tags[e] = NUPS_INVALID_KEY;
        __syncthreads();
    }
    // Windows are visited in an order that interleaves the workers' chunks: the window range is cut
    // into R stretches of `per` windows; without the tier, slot u of the schedule is window
    // (u mod R) * per + u / R, so warps that run at the same time add to different replicas of a
    // hot key; with the tier, a block walks the stretch of its own worker only.
    const uint64_t W = (n + 31) / 32;
    const uint64_t per = (W + R - 1) / R;
    const uint32_t my_q = TIER == 1 ? blockIdx.x % R : 0u;
    const uint64_t team = ((uint64_t)(TIER == 1 ? blockIdx.x / R : blockIdx.x) * blockDim.x + threadIdx.x) >> 5, warp = PARTS ? team / parts : team;
    const uint32_t part = PARTS ? (uint32_t)(team - warp * parts) : 0u;            // this warp's share of the window's destinations
    const uint64_t teams = ((uint64_t)(TIER == 1 ? gridDim.x / R : gridDim.x) * blockDim.x) >> 5, nwarps = PARTS ? teams / parts : teams;
    const unsigned share = !PARTS ? 0xFFFFFFFFu : (parts == 1 ? 0xFFFFFFFFu : parts == 2 ? 0x55555555u : parts == 4 ? 0x11111111u : 0x01010101u) << part;
    const uint64_t slots = TIER == 1 ? per : per * R;
    auto window_of = [&](uint64_t u) -> uint64_t {
        if (u >= slots) return W;
        const uint64_t w = TIER == 1 ? (uint64_t)my_q * per + u : (u % R) * per + u / R;
        return (w < W) ? w : W;
    };
    auto load_key = [&](uint64_t w) -> uint32_t {
        return (w < W && w * 32 + lane < n) ? __ldg(keys + w * 32 + lane) : NUPS_INVALID_KEY;
    };
    // lookups run two windows ahead of the reductions
    uint64_t win_a = window_of(warp), win_b = window_of(warp + nwarps);
    uint32_t key_a = load_key(win_a), key_b = load_key(win_b);
    uint32_t bits_a = (HOT && key_a < v.num_keys) ? __ldg(v.hot_bits + (key_a >> 5)) : 0u;
    for (uint64_t u = warp; u < slots; u += nwarps) {
        const uint64_t win = win_a;
        const uint32_t key = key_a;
        const uint32_t bits = bits_a;
        win_a = win_b; key_a = key_b;
        bits_a = (HOT && key_a < v.num_keys) ? __ldg(v.hot_bits + (key_a >> 5)) : 0u;
        win_b = window_of(u + 2 * nwarps);
        key_b = load_key(win_b);
        if (win >= W) continue;
        const uint64_t base = win * 32;
        const uint64_t i = base + lane;
        const bool in = i < n;
        const bool valid = in && key < v.num_keys;
        if (in && !valid && part == 0) flag_bad_key(v);
        // destination: row offset in floats, lowest bit set when it lies in the replica slab
        unsigned long long dest = NO_ROW - lane;          // invalid rows: a value no other lane has
        bool hot = false;
        size_t hrow = 0;
        int tier = -1;                                    // shared-memory accumulator of this row, if any
        if (valid) {
            dest = ((unsigned long long)key * L4) << 3;
            if (HOT && ((bits >> (key & 31)) & 1u)) {
                hot = true;
                const uint32_t slot = (uint32_t)__ldg(v.slot_of + key);
                const uint32_t q = rows_per_item == 1 ? worker_of_item(i, n_items, R)
                                                      : worker_of_item(i / rows_per_item, n_items, R);
                dest = ((((unsigned long long)q * v.Hcap + slot) * L4) << 3) | 1ull;
                hrow = (size_t)q * v.Hcap + slot;
                if (TIER == 1 && slot < tier_rows && q == my_q) tier = (int)slot;
            }
            if (TIER == 2) {
                const uint32_t at = key % tier_rows;
                uint32_t owner = tags[at];
                if (owner == NUPS_INVALID_KEY) {
                    owner = atomicCAS(&tags[at], NUPS_INVALID_KEY, key);
                    if (owner == NUPS_INVALID_KEY) owner = key;
                }
                if (owner == key) tier = (int)at;
            }
        }
        if (v.count && part == 0) {
            if (valid) atomicAdd(v.cnt + key, 1ull);
            unsigned hot_m = __ballot_sync(0xFFFFFFFFu, valid && hot);
            unsigned cold_m = __ballot_sync(0xFFFFFFFFu, valid && !hot);
            if (lane == 0) {
                if (hot_m) atomicAdd(&v.st->hot_hits, (unsigned long long)__popc(hot_m));
                if (cold_m) atomicAdd(&v.st->cold_hits, (unsigned long long)__popc(cold_m));
            }
        }
        const unsigned grp = __match_any_sync(0xFFFFFFFFu, dest);
        const bool leader = valid && (lane == (unsigned)(__ffs(grp) - 1));
        // mark the slot as touched: one lane per destination, and only if nobody has yet (a hot slot would
        // otherwise take hundreds of thousands of stores to one address)
        if (HOT && leader && hot) {
            uint32_t* flag = v.dirty + hrow;          // replica row index = q * Hcap + slot
            if (*flag == 0u) *flag = 1u;
        }
        unsigned singles = __ballot_sync(0xFFFFFFFFu, leader && __popc(grp) == 1) & share;
        unsigned multis = __ballot_sync(0xFFFFFFFFu, leader && __popc(grp) > 1) & share;

        // rows that are alone in their window: PUSH_UNROLL at a time
        while (singles) {
            int src[PUSH_UNROLL], tr[PUSH_UNROLL];
            unsigned long long de[PUSH_UNROLL];
#pragma unroll
            for (int u4 = 0; u4 < PUSH_UNROLL; ++u4) {
                src[u4] = singles ? __ffs(singles) - 1 : -1;
                singles &= singles - 1;
                de[u4] = __shfl_sync(0xFFFFFFFFu, dest, src[u4] < 0 ? 0 : src[u4]);
                tr[u4] = TIER ? __shfl_sync(0xFFFFFFFFu, tier, src[u4] < 0 ? 0 : src[u4]) : -1;
            }
            if constexpr (F64) {
                // the two rows one after the other in one run of lanes: a row that does not fill its last 32 lanes leaves
                // them to the next one
                static_assert(PUSH_UNROLL == 2, "two rows share a run of lanes");
                const uint32_t both = src[1] >= 0 ? 2 * LE : LE;
                // where element 0 of the run would lie if all of it were the first row's, or the second one's
                const uint64_t from[2] = {(base + src[0]) * LE, (base + src[1]) * LE - LE};
                auto turn = [&](uint32_t e0, auto width) {
                    constexpr int W = decltype(width)::value;
                    typename E::T a[W], b[W];
#pragma unroll
                    for (int k = 0; k < W; ++k) {
                        const uint32_t e = e0 + 32 * k;
                        if (e < both) {
                            const uint64_t in_off = (e >= LE ? from[1] : from[0]) + e;
                            a[k] = E::load(A.delta, in_off);
                            if (TWO) b[k] = E::load(B.delta, in_off);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < W; ++k) {
                        const uint32_t e = e0 + 32 * k;
                        if (e < both) {
                            const unsigned long long d = e >= LE ? de[1] : de[0];
                            const bool h = HOT && (d & 1ull);
                            const uint64_t off = (d >> 3) * 2 + (e >= LE ? e - LE : e);
                            E::reduce(h ? A.slab : A.table, off, a[k]);
                            if (TWO) E::reduce(h ? B.slab : B.table, off, b[k]);
                        }
                    }
                };
                if (!PARTS && LE <= PUSH_SHORT) turn(lane, std::integral_constant<int, 2>());
                else for (uint32_t e0 = lane; e0 < both; e0 += 32 * PUSH_WIDE) turn(e0, std::integral_constant<int, PUSH_WIDE>());
                continue;
            }
            for (uint32_t c = lane; c < LE; c += 32) {
                typename E::T a[PUSH_UNROLL], b[PUSH_UNROLL];
#pragma unroll
                for (int u4 = 0; u4 < PUSH_UNROLL; ++u4) {
                    if (src[u4] >= 0) {
                        const uint64_t in_off = (base + src[u4]) * LE + c;
                        a[u4] = E::load(A.delta, in_off);
                        if (TWO) b[u4] = E::load(B.delta, in_off);
                    }
                }
#pragma unroll
                for (int u4 = 0; u4 < PUSH_UNROLL; ++u4) {
                    if (src[u4] >= 0) {
                        bool in_tier = false;
                        if constexpr (TIER != 0) {
                            in_tier = tr[u4] >= 0;
                            if (in_tier) {
                                // accumulator rows are stored component by component, [4][L4], so that the 32
                                // lanes of one addition fall into 32 different banks
                                float* t = tier_mem + (size_t)tr[u4] * L4 * 4 + c;
                                atomicAdd(t, a[u4].x); atomicAdd(t + L4, a[u4].y); atomicAdd(t + 2 * L4, a[u4].z);
                                atomicAdd(t + 3 * L4, a[u4].w);
                            }
                        }
                        if (!in_tier) {
                            const bool h = HOT && (de[u4] & 1ull);
                            const uint64_t off = (de[u4] >> 3) * (F64 ? 2 : 1) + c;
                            E::reduce(h ? A.slab : A.table, off, a[u4]);
                            if (TWO) E::reduce(h ? B.slab : B.table, off, b[u4]);
                        }
                    }
                }
            }
            if (TIER && lane == 0) {
#pragma unroll
                for (int u4 = 0; u4 < PUSH_UNROLL; ++u4)
                    if (src[u4] >= 0 && tr[u4] >= 0 && !((touched[tr[u4] >> 5] >> (tr[u4] & 31)) & 1u))
                        atomicOr(&touched[tr[u4] >> 5], 1u << (tr[u4] & 31));
            }
        }
        // destinations hit more than once in the window: sum the members (loads PUSH_UNROLL at a time), one reduction
        while (multis) {
            const int ld = __ffs(multis) - 1;
            multis &= multis - 1;
            const unsigned members = __shfl_sync(0xFFFFFFFFu, grp, ld);
            const unsigned long long de = __shfl_sync(0xFFFFFFFFu, dest, ld);
            const int tr = TIER ? __shfl_sync(0xFFFFFFFFu, tier, ld) : -1;
            const bool h = HOT && (de & 1ull);
            for (uint32_t c = lane; c < LE; c += 32) {
                typename E::T a = E::zero(), b = a;
                unsigned mm = members;
                while (mm) {
                    int m[PUSH_UNROLL];
                    typename E::T x[PUSH_UNROLL], y[PUSH_UNROLL];
#pragma unroll
                    for (int u4 = 0; u4 < PUSH_UNROLL; ++u4) {
                        m[u4] = mm ? __ffs(mm) - 1 : -1;
                        mm &= mm - 1;
                    }
#pragma unroll
                    for (int u4 = 0; u4 < PUSH_UNROLL; ++u4) {
                        if (m[u4] >= 0) {
                            const uint64_t in_off = (base + m[u4]) * LE + c;
                            x[u4] = E::load(A.delta, in_off);
                            if (TWO) y[u4] = E::load(B.delta, in_off);
                        }
                    }
#pragma unroll
                    for (int u4 = 0; u4 < PUSH_UNROLL; ++u4) {
                        if (m[u4] >= 0) {
                            a = E::add(a, x[u4]);
                            if (TWO) b = E::add(b, y[u4]);
                        }
                    }
                }
                bool in_tier = false;
                if constexpr (TIER != 0) {
                    in_tier = tr >= 0;
                    if (in_tier) {
                        float* t = tier_mem + (size_t)tr * L4 * 4 + c;
                        atomicAdd(t, a.x); atomicAdd(t + L4, a.y); atomicAdd(t + 2 * L4, a.z); atomicAdd(t + 3 * L4, a.w);
                    }
                }
                if (!in_tier) {
                    const uint64_t off = (de >> 3) * (F64 ? 2 : 1) + c;
                    E::reduce(h ? A.slab : A.table, off, a);
                    if (TWO) E::reduce(h ? B.slab : B.table, off, b);
                }
            }
            if (TIER && tr >= 0 && lane == 0 && !((touched[tr >> 5] >> (tr & 31)) & 1u))
                atomicOr(&touched[tr >> 5], 1u << (tr & 31));
        }
    }
    if (TIER) {
        // hand the block's sums to the worker's replica: one reduction per touched row
        __syncthreads();
        for (uint32_t sl = threadIdx.x >> 5; sl < tier_rows; sl += blockDim.x >> 5) {
            if (!((touched[sl >> 5] >> (sl & 31)) & 1u)) continue;
            float* dst = TIER == 2 ? A.table + (size_t)tags[sl] * L4 * 4 : A.slab + ((size_t)my_q * v.Hcap + sl) * L4 * 4;
            const float* t = tier_mem + (size_t)sl * L4 * 4;
            for (uint32_t c = lane; c < L4; c += 32)
                red_add_v4(dst + (size_t)c * 4, make_float4(t[c], t[c + L4], t[c + 2 * L4], t[c + 3 * L4]));
        }
    }
}

// ---------------------------------------------------------------------------------------------
// push, deterministic mode: the rows of one destination are added one by one in input order.  A destination is one
// number: the key, or num_keys + worker * H + slot for a replica row; num_keys + R * H marks a bad key.
// Measured: 200,003 rows of 64 floats (Zipf 0.9 over 2M keys, 1,000 of them replicated) 430 -> 96 us with the merge: keys
// 14, three sort passes 36, push_apply_kernel 28, push_chain_kernel 10 us.
//   n <= SMALL_PUSH_ROWS: one launch without any sorting (push_small_kernel).
//   else: the rows are sorted stably by destination (nups_sort.cuh), push_apply_kernel adds the rows of every destination
//   that has at most APPLY_ROWS of them, and push_chain_kernel those of the few that have more.
// ---------------------------------------------------------------------------------------------
template <class K, bool HOT>
struct PushDest {
    View v;
    const uint32_t* keys;
    uint64_t n_items;
    uint32_t rows_per_item;
    bool note;                  // count the accesses, flag bad keys, mark the replicas as touched

    __device__ __forceinline__ K invalid() const { return (K)v.num_keys + (K)((uint64_t)v.R * v.H); }
    // rows i, i + step, ...; called by whole warps.  The lookups of the rows go side by side: each is a chain of up to three
    // dependent loads.
    template <int N>
    __device__ __forceinline__ void operator()(uint64_t i, uint64_t step, uint64_t n, K (&d)[N]) const
    {
        uint32_t key[N], bits[N], slot[N];
#pragma unroll
        for (int m = 0; m < N; ++m) key[m] = i + m * step < n ? __ldg(keys + i + m * step) : 0u;
#pragma unroll
        for (int m = 0; m < N; ++m) bits[m] = HOT && key[m] < v.num_keys ? __ldg(v.hot_bits + (key[m] >> 5)) >> (key[m] & 31) & 1u : 0u;
#pragma unroll
        for (int m = 0; m < N; ++m) slot[m] = HOT && bits[m] ? (uint32_t)__ldg(v.slot_of + key[m]) : 0u;
        uint32_t* flag[N];
        bool clean[N];
#pragma unroll
        for (int m = 0; m < N; ++m) {
            const uint64_t row = i + m * step;
            const bool valid = row < n && key[m] < v.num_keys;
            d[m] = valid ? (K)key[m] : invalid();
            flag[m] = nullptr;
            if (HOT && valid && bits[m]) {
                const uint32_t q = worker_of_item(rows_per_item == 1 ? row : row / rows_per_item, n_items, v.R);
                d[m] = (K)v.num_keys + (K)((uint64_t)q * v.H + slot[m]);
                flag[m] = v.dirty + (size_t)q * v.Hcap + slot[m];
            }
            clean[m] = note && flag[m] && *flag[m] == 0u;
        }
#pragma unroll
        for (int m = 0; m < N; ++m) {
            const bool in = i + m * step < n, valid = in && key[m] < v.num_keys, hot = flag[m] != nullptr;
            if (clean[m]) *flag[m] = 1u;
            if (note && in && !valid) flag_bad_key(v);
            if (note && v.count) {
                if (valid) atomicAdd(v.cnt + key[m], 1ull);
                const unsigned hot_m = __ballot_sync(0xFFFFFFFFu, hot);
                const unsigned cold_m = __ballot_sync(0xFFFFFFFFu, valid && !hot);
                if ((threadIdx.x & 31) == 0) {
                    if (hot_m) atomicAdd(&v.st->hot_hits, (unsigned long long)__popc(hot_m));
                    if (cold_m) atomicAdd(&v.st->cold_hits, (unsigned long long)__popc(cold_m));
                }
            }
        }
    }
};

// first 16-byte chunk of a destination's row in the value (which = 0) or accumulator table
template <class K>
__device__ __forceinline__ float4* dest_row(const View& v, K d, int which)
{
    if (d < (K)v.num_keys) return (float4*)(which ? v.acc : v.val) + (uint64_t)d * v.L4;
    const K r = d - (K)v.num_keys, q = r / (K)v.H, slot = r - q * (K)v.H;
    return (float4*)(which ? v.dacc : v.dval) + ((uint64_t)q * v.Hcap + slot) * v.L4;
}

constexpr uint32_t APPLY_ROWS = 32;          // destinations with more rows than this go to push_chain_kernel
constexpr unsigned APPLY_THREADS = 256;

// A warp takes the destinations that begin in its window of sorted positions.  W lanes serve one destination (rows of up to
// 16 chunks leave half a warp or more idle otherwise), each group of lanes works on two destinations at a time: most
// destinations have one or two rows, so what counts is how many row fetches are outstanding.  The window is short enough
// that a group of lanes has at most four such pairs to take one after the other.  (Lanes of their own for every position,
// whether a destination begins there or not, hide latency better but take 2.5 times the instructions: 54 us instead of
// 37 us for 200,000 rows of 64 floats.)
template <int W> constexpr unsigned APPLY_WINDOW = 4 * 2 * 32 / W;

template <class K, bool F64, int W>
__global__ void __launch_bounds__(APPLY_THREADS, 4)
push_apply_kernel(View v, const K* __restrict__ dest, const uint32_t* __restrict__ idx, uint64_t n64, K invalid,
                  const float4* __restrict__ dv, const float4* __restrict__ da, uint32_t* __restrict__ longs,
                  uint32_t* __restrict__ long_count)
{
    grid_dependency_wait();
    constexpr unsigned FULL = 0xFFFFFFFFu;
    constexpr int GROUPS = 32 / W, U = 2;
    constexpr unsigned WIN = APPLY_WINDOW<W>;
    static_assert(WIN <= 32, "a window is looked at by one warp");
    __shared__ uint32_t s_idx[APPLY_THREADS / 32][WIN];
    __shared__ K s_dest[APPLY_THREADS / 32][WIN];
    __shared__ uint8_t s_begin[APPLY_THREADS / 32][WIN];           // where the window's destinations begin, in order
    const unsigned lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const uint64_t base64 = (((uint64_t)blockIdx.x * APPLY_THREADS + threadIdx.x) >> 5) * WIN;
    if (base64 >= n64) return;
    const uint32_t base = (uint32_t)base64, n = (uint32_t)n64;     // positions fit 32 bits; sums with a window may not
    const bool look = lane < WIN, in = look && base64 + lane < n64;
    const K d = in ? dest[base64 + lane] : invalid;
    K before = __shfl_up_sync(FULL, d, 1);
    if (lane == 0) before = base ? dest[base - 1] : d;
    const bool begins = look && (before != d || base64 + lane == 0);
    const unsigned bounds = __ballot_sync(FULL, begins);           // bad keys and the end of the input sort last: one run
    const unsigned nb = __popc(bounds), nh = __popc(__ballot_sync(FULL, begins && d != invalid));
    if (begins) s_begin[wib][__popc(bounds & ((1u << lane) - 1u))] = (uint8_t)lane;
    if (look) { s_idx[wib][lane] = in ? idx[base64 + lane] : 0u; s_dest[wib][lane] = d; }
    __syncwarp();
    const unsigned group = lane / W, c0 = lane % W;
    const uint32_t L4 = v.L4;
    // row numbers of the destination's rows: `at` counts from the window's first position
    auto row_at = [&](uint32_t at) -> uint64_t { return (uint64_t)(at < WIN ? s_idx[wib][at] : idx[base64 + at]) * L4; };
    for (unsigned k0 = group; k0 < nh; k0 += U * GROUPS) {
        uint32_t begin[U], end[U];
        float4* row[U];
        bool live[U];
        K to[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned k = k0 + u * GROUPS;
            live[u] = k < nh;
            begin[u] = end[u] = 0;
            to[u] = invalid;
            if (!live[u]) continue;
            begin[u] = s_begin[wib][k];
            to[u] = s_dest[wib][begin[u]];
            if (k + 1 < nb) { end[u] = s_begin[wib][k + 1]; continue; }
            uint32_t e = WIN;
            if (base64 + e < n64 && dest[base64 + e] == to[u]) {
                if (base64 + begin[u] + APPLY_ROWS < n64 && dest[base64 + begin[u] + APPLY_ROWS] == to[u]) {
                    if (c0 == 0) longs[atomicAdd(long_count, 1u)] = base + begin[u];
                    live[u] = false;
                } else {
                    while (base64 + e < n64 && dest[base64 + e] == to[u]) ++e;
                }
            }
            end[u] = min(e, n - base);
        }
#pragma unroll
        for (int which = 0; which < 2; ++which) {
            const float4* src = which ? da : dv;
            if (!src) continue;
#pragma unroll
            for (int u = 0; u < U; ++u) row[u] = live[u] ? dest_row<K>(v, to[u], which) : nullptr;
            for (uint32_t c = c0; c < L4; c += W) {
                float4 a[U], x[U];
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (live[u]) { a[u] = row[u][c]; x[u] = ld_stream_v4(src + row_at(begin[u]) + c); }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (!live[u]) continue;
                    a[u] = add_chunk<F64>(a[u], x[u]);
                    for (uint32_t at = begin[u] + 1; at < end[u]; at += 4) {       // loads issued together, additions kept in order
                        float4 y[4];
#pragma unroll
                        for (int m = 0; m < 4; ++m)
                            if (at + m < end[u]) y[m] = ld_stream_v4(src + row_at(at + m) + c);
#pragma unroll
                        for (int m = 0; m < 4; ++m)
                            if (at + m < end[u]) a[u] = add_chunk<F64>(a[u], y[m]);
                    }
                    row[u][c] = a[u];
                }
            }
        }
    }
}

// Destinations with many rows (a frequent key): a chain of dependent additions per value, which only the columns can
// share out.  One block takes one group of 32 values of the row (CH chunks of 16 bytes).  Four warps bring the rows' parts
// into a ring in shared memory by asynchronous copies, five stages ahead; lane l of the fifth adds up value l.  Fetched by
// plain loads, four rows at a time, the chain would wait for memory at every fourth row.  Measured: 290,000 rows of 128 floats,
// 93,000 of them of one key: 24.8 ms with plain loads, 0.65 ms (6 ns a row; the additions alone need about 2).
constexpr unsigned CHAIN_THREADS = 160, CHAIN_STAGES = 6, CHAIN_STAGE_BYTES = 8192;
constexpr unsigned CHAIN_SMEM = CHAIN_STAGES * CHAIN_STAGE_BYTES;  // 48 KB: four blocks per multiprocessor

// The copying warps and the adding warp meet here, at different places of the kernel, once per stage.
__device__ __forceinline__ void chain_stage_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(CHAIN_THREADS) : "memory"); }

template <class K, bool F64>
__global__ void __launch_bounds__(CHAIN_THREADS)
push_chain_kernel(View v, const K* __restrict__ dest, const uint32_t* __restrict__ idx, uint64_t n,
                  const float4* __restrict__ dv, const float4* __restrict__ da, const uint32_t* __restrict__ longs,
                  const uint32_t* __restrict__ long_count)
{
    grid_dependency_wait();
    using V = typename std::conditional<F64, double, float>::type;
    constexpr unsigned FULL = 0xFFFFFFFFu;
    constexpr uint32_t CH = 32 * sizeof(V) / 16;                   // chunks of a column group
    constexpr uint32_t ROWS = CHAIN_STAGE_BYTES / (CH * 16);       // rows per stage
    constexpr uint32_t COPIES = ROWS * CH / 128;                   // 16-byte copies per producing thread and stage
    constexpr uint32_t LOOK = 4;                                   // stages whose row numbers are looked up at once
    extern __shared__ __align__(16) unsigned char ring[];
    const unsigned lane = threadIdx.x & 31;
    const bool adds = threadIdx.x < 32;
    const uint32_t L4 = v.L4, cgroups = (L4 + CH - 1) / CH, tables = (dv ? 1u : 0u) + (da ? 1u : 0u);
    const uint64_t units = (uint64_t)*long_count * cgroups * tables;
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
    for (uint64_t unit = blockIdx.x; unit < units; unit += gridDim.x) {
        const uint32_t cg = (uint32_t)(unit % cgroups);
        const int which = (!dv || (unit / cgroups) % tables) ? 1 : 0;
        const uint64_t begin = longs[unit / cgroups / tables];
        const K d = dest[begin];
        uint64_t lo = begin, hi = n;                               // last position known to be of d, first known not to be
        while (hi - lo > 1) {
            const uint64_t step = (hi - lo + 32) / 33, at = lo + (lane + 1) * step;
            const unsigned cnt = __popc(__ballot_sync(FULL, at < hi && dest[at] == d));
            lo += cnt * step;
            hi = min(hi, lo + step);
        }
        const uint32_t rows = (uint32_t)(lo + 1 - begin), stages = (rows + ROWS - 1) / ROWS;
        const uint32_t* my_rows = idx + begin;
        // producing thread t copies chunk t % CH of rows t / CH, t / CH + 128 / CH, ... of a stage
        const uint32_t t = threadIdx.x - 32, first_row = t / CH, chunk = cg * CH + t % CH;
        const float4* src = (which ? da : dv) + chunk;
        auto look_up = [&](uint32_t stage, uint32_t (&r)[LOOK * COPIES]) {
#pragma unroll
            for (uint32_t k = 0; k < LOOK * COPIES; ++k) {
                const uint32_t row = stage * ROWS + first_row + k * (128 / CH);
                r[k] = row < rows && chunk < L4 ? __ldg(my_rows + row) : 0xFFFFFFFFu;
            }
        };
        const uint32_t col = cg * 32 + lane;                       // the value this lane adds up
        const bool mine = adds && col < L4 * (16 / sizeof(V));
        V* out = reinterpret_cast<V*>(dest_row<K>(v, d, which)) + col;
        V acc = mine ? *out : V(0);
        if (!adds) {
            uint32_t r[LOOK * COPIES], ahead[LOOK * COPIES];       // row numbers of LOOK stages, and of the LOOK after them
            look_up(0, r);
            for (uint32_t stage0 = 0; stage0 < stages + CHAIN_STAGES - 1; stage0 += LOOK) {
                look_up(stage0 + LOOK, ahead);
#pragma unroll
                for (uint32_t l = 0; l < LOOK; ++l) {
                    const uint32_t stage = stage0 + l;
                    if (stage >= CHAIN_STAGES - 1 && stage < stages + CHAIN_STAGES - 1) {
                        asm volatile("cp.async.wait_group %0;" ::"n"(CHAIN_STAGES - 2) : "memory");
                        chain_stage_barrier();                     // stage - (CHAIN_STAGES - 1) is there, the one before it added up
                    }
                    const uint32_t to = ring_s + stage % CHAIN_STAGES * CHAIN_STAGE_BYTES + t * 16;
#pragma unroll
                    for (uint32_t k = 0; k < COPIES; ++k)
                        if (r[l * COPIES + k] != 0xFFFFFFFFu)
                            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + k * 2048), "l"(src + (uint64_t)r[l * COPIES + k] * L4) : "memory");
                    asm volatile("cp.async.commit_group;" ::: "memory");
                }
#pragma unroll
                for (uint32_t k = 0; k < LOOK * COPIES; ++k) r[k] = ahead[k];
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        if (adds)
        for (uint32_t stage = 0; stage < stages; ++stage) {
            chain_stage_barrier();
            const V* x = reinterpret_cast<const V*>(ring + stage % CHAIN_STAGES * CHAIN_STAGE_BYTES) + lane;
            const uint32_t left = min(rows - stage * ROWS, ROWS);
            uint32_t r = 0;
            if (left == ROWS) {
                constexpr uint32_t B = 16;                         // the next rows leave shared memory while these are added
                V y[2][B];
#pragma unroll
                for (uint32_t k = 0; k < B; ++k) y[0][k] = x[k * 32];
#pragma unroll
                for (uint32_t b = 0; b < ROWS / B; ++b) {
                    if (b + 1 < ROWS / B) {
#pragma unroll
                        for (uint32_t k = 0; k < B; ++k) y[(b + 1) & 1][k] = x[((b + 1) * B + k) * 32];
                    }
#pragma unroll
                    for (uint32_t k = 0; k < B; ++k) acc += y[b & 1][k];
                }
                r = ROWS;
            }
            for (; r + 8 <= left; r += 8) {
                V y[8];
#pragma unroll
                for (uint32_t k = 0; k < 8; ++k) y[k] = x[(r + k) * 32];
#pragma unroll
                for (uint32_t k = 0; k < 8; ++k) acc += y[k];
            }
            for (; r < left; ++r) acc += x[r * 32];
        }
        __syncthreads();
        if (mine) *out = acc;
    }
}

// Few rows: every block works out all rows' destinations (into shared memory), a warp per row looks whether an earlier row
// has the same destination and, if none has, finds the later ones by scanning, 128 rows at a step, and adds them in order;
// the first of its rows and the stored row move towards L2 meanwhile.
// One launch in place of seven; the scans grow with n^2.  Measured with the merge: 100 rows 7.2 us, 3,000 rows of 64 floats 18.3 to
// 24.1 us by their skew (23.5 to 30.4 with scans of 32 rows and nothing asked for ahead).  The line lies below where any skew
// makes the sort and what follows it the faster way: this kernel / the sort take, for uniform keys and for Zipf 1.4 with 1,000 keys
// replicated, 18.3 / 28.8 and 24.6 / 33.0 us at 3,072 rows of 64 floats, 20.2 / 30.9 and 31.2 / 36.3 of 256 floats; at 4,096 rows
// 22.2 / 29.4 and 34.2 / 33.4, 24.4 / 32.1 and 44.9 / 37.7; at 5,000 30.6 / 30.4 and 40.6 / 34.8, 33.2 / 33.2 and 53.6 / 39.5.
constexpr uint32_t SMALL_PUSH_ROWS = 3072;
constexpr unsigned SMALL_THREADS = 256, SMALL_LIST = 512;
static_assert(SMALL_PUSH_ROWS <= 65536, "row numbers are kept in 16 bits");
static_assert(SMALL_PUSH_ROWS % 128 == 0, "whole steps of the scans");

template <bool HOT, bool F64>
__global__ void __launch_bounds__(SMALL_THREADS)
push_small_kernel(PushDest<uint32_t, HOT> source, uint32_t n, const float4* __restrict__ dv, const float4* __restrict__ da)
{
    grid_dependency_wait();
    constexpr unsigned FULL = 0xFFFFFFFFu;
    constexpr int U = 16;                                          // rows in flight
    __shared__ __align__(16) uint32_t dest[SMALL_PUSH_ROWS];
    __shared__ uint16_t list[SMALL_THREADS / 32][SMALL_LIST];
    const View& v = source.v;
    const uint32_t L4 = v.L4, invalid = source.invalid();
    const uint32_t lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    source.note = blockIdx.x == 0;
    for (uint32_t b = 0; b < n; b += 4 * SMALL_THREADS) {
        uint32_t d[4];
        source(b + threadIdx.x, SMALL_THREADS, n, d);
#pragma unroll
        for (int m = 0; m < 4; ++m)
            if (b + threadIdx.x + m * SMALL_THREADS < n) dest[b + threadIdx.x + m * SMALL_THREADS] = d[m];
    }
    if (threadIdx.x < (0u - n) % 128u) dest[n + threadIdx.x] = 0xFFFFFFFFu;         // up to a whole step: no destination
    __syncthreads();
    const uint4* dest4 = reinterpret_cast<const uint4*>(dest);     // lane l of a step looks at rows 4 l ... 4 l + 3
    const uint32_t nwarps = gridDim.x * (SMALL_THREADS / 32);
    for (uint32_t i = (blockIdx.x * SMALL_THREADS + threadIdx.x) >> 5; i < n; i += nwarps) {
        const uint32_t d = dest[i];
        if (d == invalid) continue;
        bool first = true;
        for (uint32_t b = 0; b < i && first; b += 128) {
            const uint4 x = dest4[b / 4 + lane];
            const uint32_t j = b + 4 * lane;
            first = !__any_sync(FULL, (x.x == d && j < i) || (x.y == d && j + 1 < i) || (x.z == d && j + 2 < i) || (x.w == d && j + 3 < i));
        }
        if (!first) continue;
        for (uint32_t c = 8 * lane; c < L4; c += 256) {
            if (dv) { prefetch_l2(dv + (uint64_t)i * L4 + c); prefetch_l2(dest_row<uint32_t>(v, d, 0) + c); }
            if (da) { prefetch_l2(da + (uint64_t)i * L4 + c); prefetch_l2(dest_row<uint32_t>(v, d, 1) + c); }
        }
        // its rows, up to SMALL_LIST at a time
        for (uint32_t b = i & ~127u; b < n;) {
            uint32_t got = 0;
            for (; b < n && got + 128 <= SMALL_LIST; b += 128) {
                const uint4 x = dest4[b / 4 + lane];
                const uint32_t j = b + 4 * lane;
                // j + k < i: an earlier row, which the search above has shown to be another's
                const unsigned mine = (x.x == d ? 1u : 0u) | (x.y == d ? 2u : 0u) | (x.z == d ? 4u : 0u) | (x.w == d ? 8u : 0u);
                if (!__any_sync(FULL, mine != 0u)) continue;
                uint32_t at = got;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const unsigned m = __ballot_sync(FULL, (mine >> k) & 1u);
                    at += __popc(m & ((1u << lane) - 1u));
                    got += __popc(m);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if ((mine >> k) & 1u) list[wib][at++] = (uint16_t)(j + k);
            }
            __syncwarp();
#pragma unroll
            for (int which = 0; which < 2; ++which) {
                const float4* src = which ? da : dv;
                if (!src) continue;
                if (got > U)                                       // a chain: all of its rows start towards L2
                    for (uint32_t e = lane; e < got; e += 32)
                        for (uint32_t c = 0; c < L4; c += 8) prefetch_l2(src + (uint64_t)list[wib][e] * L4 + c);
                float4* row = dest_row<uint32_t>(v, d, which);
                for (uint32_t c = lane; c < L4; c += 32) {
                    float4 a = row[c];
                    for (uint32_t e = 0; e < got; e += U) {
                        float4 x[U];
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (e + u < got) x[u] = ld_stream_v4(src + (uint64_t)list[wib][e + u] * L4 + c);
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (e + u < got) a = add_chunk<F64>(a, x[u]);
                    }
                    row[c] = a;
                }
            }
            __syncwarp();
        }
    }
}

static int bits_for(unsigned long long maxval)
{
    int b = 1;
    while (b < 64 && (maxval >> b)) ++b;
    return b;
}

// can destinations be numbered with 32 bits?
static bool narrow_dest(const nups_store* s) { return s->num_keys + (uint64_t)s->R * s->H < 0xFFFFFFFFull; }
static unsigned long long invalid_dest(const nups_store* s) { return s->num_keys + (uint64_t)s->R * s->H; }

size_t nups_push_scratch_bytes(const nups_store* s, uint64_t n)
{
    if (!s->cfg.deterministic || (narrow_dest(s) && n <= SMALL_PUSH_ROWS)) return 0;     // push_small_kernel needs none
    const size_t key = narrow_dest(s) ? 4 : 8;
    return 2 * align256(n * key) + 2 * align256(n * 4) + align256((sort_plan(n, bits_for(invalid_dest(s))).hist_words() + 1) * 4);
}

nups_status nups_push_internal(nups_store* s, const uint32_t* d_keys, uint64_t n, uint32_t rows_per_item,
                               const float* d_dval, const float* d_dacc, cudaStream_t st)
{
    char* sc = nullptr;
    if (s->cfg.deterministic && n) {
        nups_status rc = nups_scratch(s, nups_push_scratch_bytes(s, n), &sc);
        if (rc != NUPS_OK) return rc;
    }
    return nups_push_with_scratch(s, d_keys, n, rows_per_item, d_dval, d_dacc, sc, st);
}

template <class K, bool HOT>
static nups_status push_ordered(nups_store* s, const View& v, const uint32_t* d_keys, uint64_t n, uint64_t n_items,
                                uint32_t rows_per_item, const float* d_dval, const float* d_dacc, char* sc, cudaStream_t st)
{
    const float4 *dv = (const float4*)d_dval, *da = (const float4*)d_dacc;
    const bool f64 = s->vb == 8;
    PushDest<K, HOT> source = {v, d_keys, n_items, rows_per_item, true};
    if constexpr (sizeof(K) == 4) {
        if (n <= SMALL_PUSH_ROWS) {
            const unsigned grid = grid_for(n, SMALL_THREADS / 32, (unsigned)s->sm_count * 4);
            if (f64) nups_launch_dependent(push_small_kernel<HOT, true>, grid, SMALL_THREADS, 0, st, source, (uint32_t)n, dv, da);
            else nups_launch_dependent(push_small_kernel<HOT, false>, grid, SMALL_THREADS, 0, st, source, (uint32_t)n, dv, da);
            LAUNCH_CHECK(s);
            return NUPS_OK;
        }
    }
    const K invalid = (K)invalid_dest(s);
    const SortPlan plan = sort_plan(n, bits_for(invalid));
    K* k0 = (K*)sc; sc += align256(n * sizeof(K));
    K* k1 = (K*)sc; sc += align256(n * sizeof(K));
    uint32_t* v0 = (uint32_t*)sc; sc += align256(n * 4);
    uint32_t* v1 = (uint32_t*)sc; sc += align256(n * 4);
    uint32_t* hist = (uint32_t*)sc;
    nups_launch_dependent(sort_begin_kernel<K, PushDest<K, HOT>>, plan.tiles, SORT_THREADS, 0, st, source, k0, hist, plan);
    LAUNCH_CHECK(s);
    K* dest;
    uint32_t* idx;
    nups_status rc = sort_passes<K>(s, k0, v0, k1, v1, hist, plan, st, &dest, &idx);
    if (rc != NUPS_OK) return rc;
    uint32_t* longs = (uint32_t*)(dest == k0 ? k1 : k0);           // the other key buffer is free now
    uint32_t* long_count = hist + plan.hist_words();
#define NUPS_APPLY(F64_, W_)                                                                                              \
    nups_launch_dependent(push_apply_kernel<K, F64_, W_>, grid_for(n, APPLY_THREADS / 32 * APPLY_WINDOW<W_>), APPLY_THREADS, 0, st, v, (const K*)dest, (const uint32_t*)idx, n, \
                          invalid, dv, da, longs, long_count)
    if (f64) { if (v.L4 <= 8) NUPS_APPLY(true, 8); else if (v.L4 <= 16) NUPS_APPLY(true, 16); else NUPS_APPLY(true, 32); }
    else { if (v.L4 <= 8) NUPS_APPLY(false, 8); else if (v.L4 <= 16) NUPS_APPLY(false, 16); else NUPS_APPLY(false, 32); }
#undef NUPS_APPLY
    LAUNCH_CHECK(s);
    const unsigned chains = (unsigned)s->sm_count * 4;             // 48 KB of shared memory each: four per multiprocessor
    if (n > APPLY_ROWS) {
        if (f64) nups_launch_dependent(push_chain_kernel<K, true>, chains, CHAIN_THREADS, CHAIN_SMEM, st, v, (const K*)dest, (const uint32_t*)idx, n, dv, da, (const uint32_t*)longs, (const uint32_t*)long_count);
        else nups_launch_dependent(push_chain_kernel<K, false>, chains, CHAIN_THREADS, CHAIN_SMEM, st, v, (const K*)dest, (const uint32_t*)idx, n, dv, da, (const uint32_t*)longs, (const uint32_t*)long_count);
        LAUNCH_CHECK(s);
    }
    return NUPS_OK;
}

nups_status nups_push_with_scratch(nups_store* s, const uint32_t* d_keys, uint64_t n, uint32_t rows_per_item,
                                   const float* d_dval, const float* d_dacc, char* sc, cudaStream_t st)
{
    if (n == 0 || (!d_dval && !d_dacc)) return NUPS_OK;
    View v = nups_view(s);
    uint64_t n_items = n / rows_per_item;
    if (!s->cfg.deterministic) {
        const bool two = d_dval && d_dacc;
        const unsigned blocks = (unsigned)s->sm_count * (two ? PUSH_BLOCKS - 1 : PUSH_BLOCKS);
        PushPair V = {(const float4*)d_dval, s->val, s->dval};
        PushPair C = {(const float4*)d_dacc, s->acc, s->dacc};
        PushPair A = d_dval ? V : C, B = C;
        // shared-memory tier: single-table calls with replicated keys, enough blocks to give every worker some
        uint32_t tier_rows = 0;
        size_t tier_bytes = 0;
        const bool cache = !s->H && !two && n >= 32768 && s->vb == 4;  // no replicated keys: accumulators as a row cache
        // (with the row cache, more blocks cost more accumulators to fill and to hand over than they save: 40,000 rows 17 -> 19 us)
        const uint32_t parts = cache ? 1 : window_parts(n, (uint64_t)blocks * (PUSH_THREADS / 32), 8);
        unsigned grid = grid_for(n * parts, PUSH_THREADS, blocks);                 // resident at once, grid-stride
        if ((s->H && !two && rows_per_item == 1 && grid >= s->R && n >= 32768 && s->vb == 4) || cache) {
            const size_t row_bytes = (size_t)s->L * 4;
            size_t budget = (size_t)(192 / PUSH_BLOCKS) * 1024;                 // the blocks of a multiprocessor share 192 KB
            const size_t per_row = row_bytes + (cache ? 4 : 0) + 1;    // sums, owner tag, touched bit (rounded up)
            tier_rows = s->cfg.smem_hot_rows ? s->cfg.smem_hot_rows : (uint32_t)(budget / per_row);
            if (tier_rows > budget / per_row) tier_rows = (uint32_t)(budget / per_row);
            if (cache && tier_rows > 1024) tier_rows = 1024;
            if (!cache && tier_rows > s->H) tier_rows = (uint32_t)s->H;
            tier_bytes = tier_rows * row_bytes + ((tier_rows + 31) / 32) * 4 + (cache ? tier_rows * 4 : 0);
            if (tier_rows && !s->push_smem_opted) {
                CK(cudaFuncSetAttribute(push_atomic_kernel<true, false, 1, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)(budget + 2048)));
                CK(cudaFuncSetAttribute(push_atomic_kernel<true, false, 1, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)(budget + 2048)));
                CK(cudaFuncSetAttribute(push_atomic_kernel<false, false, 2, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)(budget + 2048)));
                s->push_smem_opted = true;
            }
        }
        nups_time_begin(s, st, NUPS_TIMED_PUSH);
        if (tier_rows && cache) {
            nups_launch_dependent(push_atomic_kernel<false, false, 2, false, false>, grid, PUSH_THREADS, tier_bytes, st, v, d_keys, n, A, B, n_items, rows_per_item,
                                                                             tier_rows, parts);
        } else if (tier_rows) {
            grid = grid / s->R * s->R;              // every worker gets the same number of blocks
            nups_launch_dependent(parts > 1 ? push_atomic_kernel<true, false, 1, false, true> : push_atomic_kernel<true, false, 1, false, false>, grid, PUSH_THREADS, tier_bytes, st, v, d_keys, n, A, B, n_items, rows_per_item,
                                                                             tier_rows, parts);
        } else {
#define NUPS_PUSH0(HOT_, TWO_, F64_) \
    nups_launch_dependent(parts > 1 ? push_atomic_kernel<HOT_, TWO_, 0, F64_, true> : push_atomic_kernel<HOT_, TWO_, 0, F64_, false>, grid, PUSH_THREADS, 0, st, v, d_keys, n, A, B, n_items, \
                          rows_per_item, 0, parts)
            if (s->vb == 8) {
                if (s->H) { if (two) NUPS_PUSH0(true, true, true); else NUPS_PUSH0(true, false, true); }
                else { if (two) NUPS_PUSH0(false, true, true); else NUPS_PUSH0(false, false, true); }
            } else if (s->H) {
                if (two) NUPS_PUSH0(true, true, false); else NUPS_PUSH0(true, false, false);
            } else {
                if (two) NUPS_PUSH0(false, true, false); else NUPS_PUSH0(false, false, false);
            }
#undef NUPS_PUSH0
        }
        nups_time_end(s, st);
        LAUNCH_CHECK(s);
        return NUPS_OK;
    }
    if (narrow_dest(s)) return s->H ? push_ordered<uint32_t, true>(s, v, d_keys, n, n_items, rows_per_item, d_dval, d_dacc, sc, st)
                                    : push_ordered<uint32_t, false>(s, v, d_keys, n, n_items, rows_per_item, d_dval, d_dacc, sc, st);
    return s->H ? push_ordered<unsigned long long, true>(s, v, d_keys, n, n_items, rows_per_item, d_dval, d_dacc, sc, st)
                : push_ordered<unsigned long long, false>(s, v, d_keys, n, n_items, rows_per_item, d_dval, d_dacc, sc, st);
}

extern "C" nups_status nups_push2(nups_store* s, const uint32_t* d_keys, uint64_t n, const void* d_dval_,
                                  const void* d_dacc_, void* stream)
{
    const float* d_dval = (const float*)d_dval_;
    const float* d_dacc = (const float*)d_dacc_;
    if (!s || (n && !d_keys) || n >= (1ull << 32)) return NUPS_EINVAL;
    if (d_dacc && !s->acc) return NUPS_EINVAL;
    if (n && !d_dval && !d_dacc) return NUPS_EINVAL;
    return nups_push_internal(s, d_keys, n, 1, d_dval, d_dacc, (cudaStream_t)stream);
}

extern "C" nups_status nups_push(nups_store* s, const uint32_t* d_keys, uint64_t n, const void* d_delta, void* stream)
{
    if (n && !d_delta) return NUPS_EINVAL;
    return nups_push2(s, d_keys, n, d_delta, nullptr, stream);
}

// ---------------------------------------------------------------------------------------------
// sync: merge the workers' pending updates of every touched hot slot into the stored row,
// worker 0 first, and clear them and the marks.  A warp per slot reads the workers' marks with one load each,
// so only slots and replicas that were touched cost more than that.  Rows wider than a warp are divided among
// two to eight warps as long as they make at most two waves (of 32 warps per multiprocessor: the kernel takes 56 to 60 registers).
// Measured: 1,000 slots of 512 bytes and 8 workers 9.2 -> 3.6 us (before: a thread per chunk that read every mark, the marks
// cleared by a launch of its own).  All replicas of two tables of 2,000 bytes touched, launch and events included, with 1, 2
// and 4 warps per slot: 300 slots 17.6, 12.5, 10.9 us; 1,200 slots 21.4, 16.9, 18.6; 2,400 slots 31.6, 33.7, 29.2; 4,000 bytes,
// one table, 300 slots with 1 and 8: 17.5, 10.2.  20,000 slots of 1,200 bytes with 1 and 4: 11 and 33 us.  The second wave pays
// among other work: 50,000 rows of two such tables pulled, pushed and merged, 1,200 slots: 219.7 us, with one wave 222.9;
// 2,400 slots: 228.6 and 235.0.  (Held to 64 registers the kernel merges 1,000 slots of 1,024 bytes 8 us slower.)
// The next kernel of the stream waits for the merge's end before its blocks become resident, unless the caller knows that
// it is a small one: a push or a step whose blocks fill the multiprocessors runs longer when they were placed between the
// merge's.  Measured, placed between them and after them: 1M rows pushed and 1,000 slots merged, in turn, 200 and 191 us;
// ComplEx steps of three stores in turn, every 16th with a merge, 229 and 225 us each.  Skip-gram steps, whose merges are
// followed by a draw or by an event: 456.7 and 457.7 us for 64 of them.
// ---------------------------------------------------------------------------------------------
template <bool F64>
__global__ void __launch_bounds__(256)
sync_kernel(View v, const uint32_t* __restrict__ hot_keys, uint32_t per_slot, bool early_next)      // warps per slot: 1, 2, 4 or 8
{
    if (early_next) grid_dependency_wait();
    else grid_dependency_wait_alone();
    constexpr unsigned FULL = 0xFFFFFFFFu;
    constexpr int U = 4;                                     // replica rows in flight
    const uint32_t lane = threadIdx.x & 31, L4 = v.L4;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, slot = warp / per_slot;
    const uint32_t part = (uint32_t)(warp - slot * per_slot);
    const bool real = slot < v.H;
    const uint32_t key = real ? __ldg(hot_keys + slot) : 0u;
    uint32_t marks[8], touched = 0;                          // R <= 254: marks of workers 32 w ... 32 w + 31
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        marks[w] = 0u;
        if (32 * w >= v.R) continue;
        const uint32_t r = 32 * w + lane;
        const bool set = real && r < v.R && v.dirty[(size_t)r * v.Hcap + slot] != 0u;
        marks[w] = __ballot_sync(FULL, set);
        touched += __popc(marks[w]);
    }
    if (per_slot > 1) __syncthreads();                       // a slot's warps, all of one block, have read its marks
    if (!touched) return;
    if (part == 0) {
#pragma unroll
        for (int w = 0; w < 8; ++w)
            if (marks[w] >> lane & 1u) v.dirty[(size_t)(32 * w + lane) * v.Hcap + slot] = 0u;
    }
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const size_t worker_stride = (size_t)v.Hcap * L4;
#pragma unroll
    for (int which = 0; which < 2; ++which) {
        float4* table = (float4*)(which ? v.acc : v.val);
        float4* slab = (float4*)(which ? v.dacc : v.dval);
        if (!table || !slab) continue;
        for (uint32_t c = part * 32 + lane; c < L4; c += per_slot * 32) {
            float4* row = table + (uint64_t)key * L4 + c;
            const float4 old = *row;
            float4 sum = zero;
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                float4* rep = slab + 32 * w * worker_stride + slot * L4 + c;
                for (uint32_t m = marks[w]; m;) {
                    float4* at[U];
                    float4 x[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        at[u] = m ? rep + (__ffs(m) - 1) * worker_stride : nullptr;
                        m &= m - 1;
                        if (at[u]) x[u] = *at[u];
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (at[u]) { sum = add_chunk<F64>(sum, x[u]); *at[u] = zero; }
                }
            }
            if (v.merge_mean) {                              // the mean over the workers that touched the slot
                if (F64) {
                    const double2 d = as_d2(sum);
                    sum = as_f4(make_double2(__ddiv_rn(d.x, (double)touched), __ddiv_rn(d.y, (double)touched)));
                } else {
                    const float by = (float)touched;
                    sum = make_float4(__fdiv_rn(sum.x, by), __fdiv_rn(sum.y, by), __fdiv_rn(sum.z, by), __fdiv_rn(sum.w, by));
                }
            }
            *row = add_chunk<F64>(old, sum);
        }
    }
}

nups_status nups_sync_internal(nups_store* s, cudaStream_t st, bool early_next)
{
    if (s->H == 0) return NUPS_OK;        // nothing replicated: no work at all
    View v = nups_view(s);
    nups_background_begin(s, st);
    uint32_t per_slot = 1;
    while (per_slot < 8 && per_slot * 32 < v.L4 && s->H * per_slot * 2 <= (uint64_t)s->sm_count * 64) per_slot *= 2;
    if (s->vb == 8) nups_launch_dependent(sync_kernel<true>, grid_for(s->H * per_slot, 8), 256, 0, st, v, s->hot_keys, per_slot, early_next);
    else nups_launch_dependent(sync_kernel<false>, grid_for(s->H * per_slot, 8), 256, 0, st, v, s->hot_keys, per_slot, early_next);
    const cudaError_t e = cudaGetLastError();
    nups_background_end(s, st);
    if (e != cudaSuccess) return nups_cuda_fail(e, "replica merge");
    s->launches++;
    s->syncs++;
    return NUPS_OK;
}

extern "C" nups_status nups_sync(nups_store* s, void* stream)
{
    if (!s) return NUPS_EINVAL;
    return nups_sync_internal(s, (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------------------------
// access counting and hot-set selection
// ---------------------------------------------------------------------------------------------
// A block adds up the keys it meets again in shared memory: a table of COUNT_SLOTS keys and counts, a slot belonging to the
// first key that asks for it.  Frequent keys show up early, so they take slots, and thousands of additions no longer queue
// at one address; all other keys are counted by one reduction each.  (Looking for equal keys within a warp by a match
// instruction took longer than the reductions that it saved.)  Two blocks per multiprocessor.  Measured, 4M keys over 11M:
// 79 -> 47 us at Zipf 0.8, 155 -> 34 us at Zipf 1.0 (launch and events included).
constexpr unsigned COUNT_THREADS = 1024, COUNT_SLOT_BITS = 12, COUNT_SLOTS = 1u << COUNT_SLOT_BITS, COUNT_ITEMS = 4;

__global__ void __launch_bounds__(COUNT_THREADS)
count_kernel(View v, const uint32_t* __restrict__ keys, uint64_t n)
{
    __shared__ uint32_t tag[COUNT_SLOTS], count[COUNT_SLOTS];
    for (unsigned e = threadIdx.x; e < COUNT_SLOTS; e += COUNT_THREADS) { tag[e] = NUPS_INVALID_KEY; count[e] = 0u; }
    __syncthreads();
    const uint64_t step = (uint64_t)gridDim.x * COUNT_THREADS;
    for (uint64_t i = (uint64_t)blockIdx.x * COUNT_THREADS + threadIdx.x; i < n; i += COUNT_ITEMS * step) {
        uint32_t k[COUNT_ITEMS];
#pragma unroll
        for (int m = 0; m < (int)COUNT_ITEMS; ++m) k[m] = i + m * step < n ? __ldcs(keys + i + m * step) : NUPS_INVALID_KEY;
#pragma unroll
        for (int m = 0; m < (int)COUNT_ITEMS; ++m) {
            if (k[m] >= v.num_keys) {                        // the largest 32-bit number is never a key
                if (i + m * step < n) flag_bad_key(v);
                continue;
            }
            const unsigned at = (k[m] * 0x9E3779B1u) >> (32 - COUNT_SLOT_BITS);
            uint32_t owner = tag[at];
            if (owner == NUPS_INVALID_KEY) {
                owner = atomicCAS(&tag[at], NUPS_INVALID_KEY, k[m]);
                if (owner == NUPS_INVALID_KEY) owner = k[m];
            }
            if (owner == k[m]) atomicAdd(&count[at], 1u);
            else atomicAdd(v.cnt + k[m], 1ull);
        }
    }
    __syncthreads();
    for (unsigned e = threadIdx.x; e < COUNT_SLOTS; e += COUNT_THREADS)
        if (count[e]) atomicAdd(v.cnt + tag[e], (unsigned long long)count[e]);
}

extern "C" nups_status nups_count_accesses(nups_store* s, const uint32_t* d_keys, uint64_t n, void* stream)
{
    if (!s || (n && !d_keys)) return NUPS_EINVAL;
    if (n == 0) return NUPS_OK;
    count_kernel<<<grid_for(n, COUNT_THREADS, (unsigned)s->sm_count * 2), COUNT_THREADS, 0, (cudaStream_t)stream>>>(nups_view(s), d_keys, n);
    LAUNCH_CHECK(s);
    return NUPS_OK;
}

// Is p memory of the store's GPU, which a kernel may write to?  Results go anywhere else (another GPU, the host) by the copy
// call, which finds its way there or returns an error.
static bool own_memory(const nups_store* s, const void* p)
{
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice && at.device == s->device;
}

// The counts are handed out by a copy of our own: they are next to the multiprocessors in L2 when they have just been
// counted or chosen from, and reading 64 bytes per thread at once takes them out faster than the copy call (88 MB: 42 us, 50 us).
__global__ void __launch_bounds__(256)
copy_counts_kernel(const ulonglong2* __restrict__ from, ulonglong2* __restrict__ to, uint64_t n2)
{
    const uint64_t first = (uint64_t)blockIdx.x * 1024 + threadIdx.x;
    ulonglong2 x[4];
#pragma unroll
    for (int m = 0; m < 4; ++m)
        if (first + m * 256 < n2) x[m] = __ldcg(from + first + m * 256);
#pragma unroll
    for (int m = 0; m < 4; ++m)
        if (first + m * 256 < n2) __stcs(to + first + m * 256, x[m]);
}

extern "C" nups_status nups_get_counts(nups_store* s, uint64_t* d_out, void* stream)
{
    if (!s || !d_out) return NUPS_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    if (!own_memory(s, d_out) || ((uintptr_t)d_out & 15)) {  // ... or not aligned for wide stores
        CK(cudaMemcpyAsync(d_out, s->cnt, s->num_keys * 8, cudaMemcpyDeviceToDevice, st));
        return NUPS_OK;
    }
    const uint64_t n2 = s->num_keys / 2;
    if (n2) {
        copy_counts_kernel<<<grid_for(n2, 1024), 256, 0, st>>>((const ulonglong2*)s->cnt, (ulonglong2*)d_out, n2);
        LAUNCH_CHECK(s);
    }
    if (s->num_keys & 1) CK(cudaMemcpyAsync(d_out + 2 * n2, s->cnt + 2 * n2, 8, cudaMemcpyDeviceToDevice, st));
    return NUPS_OK;
}

// Choosing the hot keys.  Only the keys that are chosen are ever sorted:
//   1. one pass over the counts: their sum, their maximum, and how many lie in each of 976 bins (exact below 32, sixteen
//      bins per power of two above).  The host reads these and knows the lowest count that is chosen, or the bin it is in;
//      a bin that holds many more keys than are wanted is cut finer by further passes;
//   2. per stretch of keys, how many lie above that count and on it; their prefix sums;
//   3. the chosen keys in key order (of those on the lowest count, the first ones), and a stable sort by count.
// Measured, the 10,000 most frequent of 11M keys: 117 us of kernels (bins 41, stretches 32, prefix sums 6, chosen keys 7, sort 25),
// where a sort of all keys by count and key took 1,400.
constexpr unsigned SELECT_THREADS = 256, SELECT_BINS = 1024, SELECT_MAX_RANGES = 2048;
constexpr uint64_t SELECT_CHUNK = 8 * SELECT_THREADS, SELECT_BIN_KEYS = 65536;

struct CountStat {
    unsigned long long sum, max;
    unsigned long long bin[SELECT_BINS];
};

__device__ __forceinline__ unsigned count_bin(unsigned long long c)
{
    if (c < 32) return (unsigned)c;
    const unsigned e = 63u - (unsigned)__clzll((long long)c);
    return 32u + (e - 5u) * 16u + (unsigned)((c >> (e - 4u)) & 15u);
}
// smallest count of a bin, and how many counts it spans (as a power of two)
static unsigned long long bin_first(unsigned b) { return b < 32 ? b : (unsigned long long)(16 + (b - 32) % 16) << ((b - 32) / 16 + 1); }
static unsigned bin_shift(unsigned b) { return b < 32 ? 0 : (b - 32) / 16 + 1; }

// FIRST: sum, maximum and the bins of count_bin.  Otherwise: the counts c with first <= c, (c - first) >> shift < SELECT_BINS.
template <bool FIRST>
__global__ void __launch_bounds__(SELECT_THREADS)
count_stat_kernel(const unsigned long long* __restrict__ cnt, uint64_t n, unsigned long long first, unsigned shift,
                  CountStat* __restrict__ out)
{
    constexpr unsigned COPIES = 4;                           // lanes of a warp that meet in a bin are spread over these
    __shared__ __align__(16) unsigned h[SELECT_BINS * COPIES];
    for (unsigned e = threadIdx.x; e < SELECT_BINS * COPIES; e += SELECT_THREADS) h[e] = 0u;
    __syncthreads();
    unsigned* mine = h + threadIdx.x % COPIES;
    unsigned long long sum = 0, mx = 0;
    unsigned zeros = 0, ones = 0;                            // most keys: counted in registers
    auto take = [&](unsigned long long c) {
        if (FIRST) {
            sum += c;
            mx = c > mx ? c : mx;
            if (c == 0) ++zeros;
            else if (c == 1) ++ones;
            else atomicAdd(mine + COPIES * count_bin(c), 1u);
        } else if (c >= first && (c - first) >> shift < SELECT_BINS) {
            atomicAdd(mine + COPIES * (unsigned)((c - first) >> shift), 1u);
        }
    };
    const uint64_t pairs = n / 2, step = (uint64_t)gridDim.x * SELECT_THREADS;
    const ulonglong2* two = reinterpret_cast<const ulonglong2*>(cnt);
    for (uint64_t i = (uint64_t)blockIdx.x * SELECT_THREADS + threadIdx.x; i < pairs; i += 4 * step) {
        ulonglong2 c[4];
#pragma unroll
        for (int m = 0; m < 4; ++m)
            if (i + m * step < pairs) c[m] = two[i + m * step];
#pragma unroll
        for (int m = 0; m < 4; ++m)
            if (i + m * step < pairs) { take(c[m].x); take(c[m].y); }
    }
    if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) take(cnt[n - 1]);
    if (FIRST) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
            const unsigned long long m2 = __shfl_xor_sync(0xFFFFFFFFu, mx, o);
            mx = m2 > mx ? m2 : mx;
            zeros += __shfl_xor_sync(0xFFFFFFFFu, zeros, o);
            ones += __shfl_xor_sync(0xFFFFFFFFu, ones, o);
        }
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&out->sum, sum);
            atomicMax(&out->max, mx);
            if (zeros) atomicAdd(h, zeros);
            if (ones) atomicAdd(h + COPIES, ones);
        }
    }
    __syncthreads();
    for (unsigned e = threadIdx.x; e < SELECT_BINS; e += SELECT_THREADS) {
        const uint4 x = reinterpret_cast<const uint4*>(h)[e];
        const unsigned long long all = (unsigned long long)x.x + x.y + x.z + x.w;
        if (all) atomicAdd(&out->bin[e], all);
    }
}

// Keys of a stretch with a count above `cut` (upper half of the word) and on it (lower half).  Two words of bits per 64 keys
// say which ones have either: the even and the odd ones.
__global__ void __launch_bounds__(SELECT_THREADS)
select_count_kernel(const unsigned long long* __restrict__ cnt, uint64_t n, uint64_t range, unsigned long long cut,
                    unsigned long long* __restrict__ found, uint2* __restrict__ bits)
{
    constexpr unsigned FULL = 0xFFFFFFFFu;
    __shared__ unsigned long long total;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t first = blockIdx.x * range, last = min(first + range, n);
    unsigned above = 0, either = 0;
    for (uint64_t b = first; b < last; b += SELECT_CHUNK) {              // a stretch is a whole number of chunks
        ulonglong2 c[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {                                    // a warp looks at 256 consecutive counts
            const uint64_t i = b + warp * 256 + k * 64 + lane * 2;
            c[k] = make_ulonglong2(0, 0);
            if (i + 1 < last) c[k] = *reinterpret_cast<const ulonglong2*>(cnt + i);
            else if (i < last) c[k].x = cnt[i];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint64_t i = b + warp * 256 + k * 64 + lane * 2;
            const bool x = i < last && c[k].x >= cut, y = i + 1 < last && c[k].y >= cut;
            const uint2 w = make_uint2(__ballot_sync(FULL, x), __ballot_sync(FULL, y));
            if (lane == 0 && i < last) bits[i >> 6] = w;
            above += (x && c[k].x > cut) + (y && c[k].y > cut);
            either += x + y;
        }
    }
    unsigned long long both = (unsigned long long)above << 32 | (either - above);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) both += __shfl_xor_sync(FULL, both, o);
    if (lane == 0) atomicAdd(&total, both);
    __syncthreads();
    if (threadIdx.x == 0) found[blockIdx.x] = total;
}

// The chosen keys and their counts in key order: all keys above `cut` and the first `ties` of those on it.  `before` = for
// every stretch, the keys above (upper half) and on the cut in the stretches before it.  A thread takes 64 keys and reads
// the counts of those whose bit is set only.
__global__ void __launch_bounds__(SELECT_THREADS)
select_write_kernel(const unsigned long long* __restrict__ cnt, uint64_t n, uint64_t range, unsigned long long cut,
                    unsigned long long ties, const unsigned long long* __restrict__ before, const uint2* __restrict__ bits,
                    uint32_t* __restrict__ keys, unsigned long long* __restrict__ counts)
{
    __shared__ unsigned long long warp_sum[SELECT_THREADS / 32];
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t first = blockIdx.x * range, last = min(first + range, n);
    unsigned long long so_far = before[blockIdx.x];
    for (uint64_t b = first; b < last; b += 64 * SELECT_THREADS) {
        const uint64_t i = b + 64 * threadIdx.x;
        const uint2 w = i < last ? bits[i >> 6] : make_uint2(0u, 0u);
        auto each = [&](auto use) {                          // the thread's keys in order
            for (unsigned left = w.x | w.y; left; left &= left - 1) {
                const unsigned at = __ffs(left) - 1;
                if (w.x >> at & 1u) use(i + 2 * at, cnt[i + 2 * at]);
                if (w.y >> at & 1u) use(i + 2 * at + 1, cnt[i + 2 * at + 1]);
            }
        };
        unsigned long long mine = 0;
        each([&](uint64_t, unsigned long long c) { mine += c > cut ? 1ull << 32 : 1ull; });
        unsigned long long inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= (unsigned)o) inc += y;
        }
        __syncthreads();                                     // the round before's readers are done
        if (lane == 31) warp_sum[warp] = inc;
        __syncthreads();
        unsigned long long here = so_far + inc - mine;
        for (unsigned k = 0; k < SELECT_THREADS / 32; ++k) {
            if (k < warp) here += warp_sum[k];
            so_far += warp_sum[k];
        }
        each([&](uint64_t key, unsigned long long c) {
            const unsigned long long above = here >> 32, on = here & 0xFFFFFFFFull;
            if (c > cut || on < ties) {
                const unsigned long long at = above + (on < ties ? on : ties);
                keys[at] = (uint32_t)key;
                counts[at] = c;
            }
            here += c > cut ? 1ull << 32 : 1ull;
        });
    }
}

// sort keys of the chosen: how far a count lies below the largest one
struct BelowMax {
    const unsigned long long* counts;
    unsigned long long max_cnt;
    template <int N>
    __device__ __forceinline__ void operator()(uint64_t i, uint64_t step, uint64_t n, unsigned long long (&d)[N]) const
    {
#pragma unroll
        for (int m = 0; m < N; ++m) d[m] = i + m * step < n ? max_cnt - counts[i + m * step] : 0ull;
    }
};

__global__ void select_out_kernel(const uint32_t* __restrict__ keys, const uint32_t* __restrict__ order, uint64_t n, uint32_t* __restrict__ out)
{
    grid_dependency_wait();
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = keys[order[i]];
}

extern "C" nups_status nups_select_hot(nups_store* s, int by_topk, uint64_t param, uint32_t* d_keys_out,
                                       uint64_t* h_n_out, void* stream)
{
    if (!s || !d_keys_out || !h_n_out) return NUPS_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const uint64_t n = s->num_keys;
    *h_n_out = 0;
    const uint64_t range = ((n + SELECT_MAX_RANGES - 1) / SELECT_MAX_RANGES + SELECT_CHUNK - 1) / SELECT_CHUNK * SELECT_CHUNK;
    const unsigned ranges = (unsigned)((n + range - 1) / range);
    const size_t bits_at = align256(sizeof(CountStat)) + align256(ranges * 8 + 8) + nups_scan_scratch_bytes(ranges);
    const size_t fixed = bits_at + align256((n + 63) / 64 * 8);
    auto bytes_for = [&](uint64_t rows, const SortPlan& plan) { return fixed + align256(rows * 4) * 3 + align256(rows * 8) * 3 + align256((plan.hist_words() + 1) * 4); };
    // the most keys that can be sorted for the `param` most frequent: those above a bin, and a bin that is not cut finer
    const uint64_t wanted = by_topk ? (param < n ? param : n) : 0, bin = wanted > SELECT_BIN_KEYS ? wanted : SELECT_BIN_KEYS;
    const uint64_t most = wanted + bin < n ? wanted + bin : n;
    char* sc;
    nups_status rc = nups_scratch(s, wanted ? bytes_for(most, sort_plan(most, 64)) : fixed, &sc);
    if (rc != NUPS_OK) return rc;
    CountStat* d_stat = (CountStat*)sc;
    CountStat stat;
    const unsigned grid = grid_for(n, 8 * SELECT_THREADS, (unsigned)s->sm_count * 8);
    CK(cudaMemsetAsync(d_stat, 0, sizeof(CountStat), st));
    count_stat_kernel<true><<<grid, SELECT_THREADS, 0, st>>>(s->cnt, n, 0, 0, d_stat);
    LAUNCH_CHECK(s);
    CK(cudaMemcpyAsync(&stat, d_stat, sizeof(stat), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    const unsigned long long total = stat.sum, max_cnt = stat.max;
    if (bits_for(n - 1) + bits_for(max_cnt) > 64) return NUPS_ESTATE;        // the call's documented limit, not this method's
    // keys above `cut` are chosen, and the first `ties` of those on it; m = how many that makes, `take` of them are wanted
    unsigned long long cut = 0, ties = 0;
    uint64_t m = 0, take = 0;
    if (by_topk) {
        take = wanted;
        if (take == 0) return NUPS_OK;
        uint64_t above = 0;                                  // keys in higher bins
        unsigned b = SELECT_BINS - 1;
        while (above + stat.bin[b] < take) above += stat.bin[b--];
        unsigned long long first = bin_first(b);
        unsigned shift = bin_shift(b);
        // the bin reaches from `first` over 2^shift counts.  Cut it finer while it holds far more keys than are wanted.
        while (shift && stat.bin[b] > bin) {
            const unsigned fine = shift > 10 ? shift - 10 : 0;
            CK(cudaMemsetAsync(d_stat, 0, sizeof(CountStat), st));
            count_stat_kernel<false><<<grid, SELECT_THREADS, 0, st>>>(s->cnt, n, first, fine, d_stat);
            LAUNCH_CHECK(s);
            CK(cudaMemcpyAsync(&stat, d_stat, sizeof(stat), cudaMemcpyDeviceToHost, st));
            CK(cudaStreamSynchronize(st));
            b = (unsigned)((1ull << (shift - fine)) - 1);    // the finer bins of the old one only
            while (above + stat.bin[b] < take) above += stat.bin[b--];
            first += (unsigned long long)b << fine;
            shift = fine;
        }
        if (shift == 0) { cut = first; ties = take - above; m = take; }
        else { cut = first - 1; ties = 0; m = above + stat.bin[b]; }         // the whole bin: the sort finds the first `take`
    } else {
        // count * n > param * total, exactly: count > floor(param * total / n)
        const unsigned __int128 q = (unsigned __int128)param * total / n;
        if (q >= max_cnt) return NUPS_OK;
        cut = (unsigned long long)q;
    }
    unsigned long long* found = (unsigned long long*)(sc + align256(sizeof(CountStat)));
    auto count_found = [&]() -> nups_status {
        select_count_kernel<<<ranges, SELECT_THREADS, 0, st>>>(s->cnt, n, range, cut, found, (uint2*)(sc + bits_at));
        LAUNCH_CHECK(s);
        return nups_scan_u64(s, found, found, ranges, found + ranges, (char*)found + align256(ranges * 8 + 8), st);
    };
    if (!by_topk) {
        rc = count_found();
        if (rc != NUPS_OK) return rc;
        unsigned long long both = 0;
        CK(cudaMemcpyAsync(&both, found + ranges, 8, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        take = m = both >> 32;
        if (m == 0) return NUPS_OK;
    }
    const SortPlan plan = sort_plan(m, bits_for(max_cnt - cut));
    const size_t need = bytes_for(m, plan);
    const bool moves = need > s->scratch_bytes;              // a larger buffer: what was found is found again there
    rc = nups_scratch(s, need, &sc);
    if (rc != NUPS_OK) return rc;
    found = (unsigned long long*)(sc + align256(sizeof(CountStat)));
    if (by_topk || moves) rc = count_found();
    if (rc != NUPS_OK) return rc;
    const uint2* bits = (const uint2*)(sc + bits_at);
    sc += fixed;
    uint32_t* keys = (uint32_t*)sc; sc += align256(m * 4);
    uint32_t* v0 = (uint32_t*)sc; sc += align256(m * 4);
    uint32_t* v1 = (uint32_t*)sc; sc += align256(m * 4);
    unsigned long long* counts = (unsigned long long*)sc; sc += align256(m * 8);
    unsigned long long* k0 = (unsigned long long*)sc; sc += align256(m * 8);
    unsigned long long* k1 = (unsigned long long*)sc; sc += align256(m * 8);
    uint32_t* hist = (uint32_t*)sc;
    select_write_kernel<<<ranges, SELECT_THREADS, 0, st>>>(s->cnt, n, range, cut, ties, found, bits, keys, counts);
    LAUNCH_CHECK(s);
    const BelowMax below = {counts, max_cnt};
    nups_launch_dependent(sort_begin_kernel<unsigned long long, BelowMax>, plan.tiles, SORT_THREADS, 0, st, below, k0, hist, plan);
    LAUNCH_CHECK(s);
    unsigned long long* sorted;
    uint32_t* order;
    rc = sort_passes<unsigned long long>(s, k0, v0, k1, v1, hist, plan, st, &sorted, &order);
    if (rc != NUPS_OK) return rc;
    uint32_t* out = own_memory(s, d_keys_out) ? d_keys_out : order == v0 ? v1 : v0;
    nups_launch_dependent(select_out_kernel, grid_for(take, 256), 256, 0, st, keys, order, take, out);
    LAUNCH_CHECK(s);
    if (out != d_keys_out) CK(cudaMemcpyAsync(d_keys_out, out, take * 4, cudaMemcpyDeviceToDevice, st));
    CK(cudaStreamSynchronize(st));
    *h_n_out = take;
    return NUPS_OK;
}

// ---------------------------------------------------------------------------------------------
// per-key management
// ---------------------------------------------------------------------------------------------
// REPLICATE, pass 1: every listed key that is not hot yet is claimed by its first list position.
// slot_of holds: >= 0 hot slot; -1 single; <= -2 a claim by list position p encoded as -(p + 2).
__global__ void claim_kernel(int* slot_of, uint64_t num_keys, const uint32_t* __restrict__ keys, uint64_t n, DevStat* st)
{
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t k = keys[i];
    if (k >= num_keys) { atomicCAS(&st->status, 0, NUPS_EKEY); return; }
    int mine = -(int)(i + 2);
    int cur = slot_of[k];
    while (cur < 0 && (cur == -1 || cur < mine)) {          // smaller position = larger (closer to -2) code
        int prev = atomicCAS(&slot_of[k], cur, mine);
        if (prev == cur) break;
        cur = prev;
    }
}
__global__ void winner_flag_kernel(const int* __restrict__ slot_of, uint64_t num_keys, const uint32_t* __restrict__ keys,
                                   uint64_t n, unsigned long long* __restrict__ flag)
{
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t k = keys[i];
    flag[i] = (k < num_keys && slot_of[k] == -(int)(i + 2)) ? 1ull : 0ull;
}
__global__ void assign_slots_kernel(int* slot_of, uint32_t* hot_bits, uint32_t* hot_keys, const uint32_t* __restrict__ keys,
                                    uint64_t n, const unsigned long long* __restrict__ flag,
                                    const unsigned long long* __restrict__ pos, uint64_t H_old)
{
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || !flag[i]) return;
    uint32_t k = keys[i];
    uint64_t slot = H_old + pos[i];
    slot_of[k] = (int)slot;
    hot_keys[slot] = k;
    atomicOr(&hot_bits[k >> 5], 1u << (k & 31));
}
// SINGLE: drop the listed keys, then renumber the surviving slots in their old order.
__global__ void demote_kernel(int* slot_of, uint32_t* hot_bits, uint64_t num_keys, const uint32_t* __restrict__ keys,
                              uint64_t n, DevStat* st)
{
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t k = keys[i];
    if (k >= num_keys) { atomicCAS(&st->status, 0, NUPS_EKEY); return; }
    slot_of[k] = -1;
    atomicAnd(&hot_bits[k >> 5], ~(1u << (k & 31)));
}
__global__ void alive_flag_kernel(const int* __restrict__ slot_of, const uint32_t* __restrict__ hot_keys, uint64_t H,
                                  unsigned long long* __restrict__ flag)
{
    uint64_t sl = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (sl >= H) return;
    flag[sl] = slot_of[hot_keys[sl]] >= 0 ? 1ull : 0ull;
}
__global__ void renumber_kernel(int* slot_of, const uint32_t* __restrict__ hot_keys, uint32_t* __restrict__ hot_keys_new,
                                uint64_t H, const unsigned long long* __restrict__ flag,
                                const unsigned long long* __restrict__ pos)
{
    uint64_t sl = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (sl >= H || !flag[sl]) return;
    uint32_t k = hot_keys[sl];
    slot_of[k] = (int)pos[sl];
    hot_keys_new[pos[sl]] = k;
}

// Shorter lists take fewer launches.  REPLICATE, up to a million keys: a block counts its winners, then every block adds up
// the counts before its own and hands out the slots.  SINGLE, up to 16,384 slots: one block finds the survivors and moves
// them up in place (a round's entries are read before any is written, and none is written beyond the entries read); with
// more of them one multiprocessor's random accesses take longer than the launches.  Measured, 10,000 keys: 25 -> 10 us (REPLICATE;
// 26 us in one block), 25 -> 13 us (SINGLE).
constexpr uint64_t ASSIGN_LIST_KEYS = 1u << 20, SMALL_LIST_KEYS = 16384;
constexpr unsigned MANAGE_THREADS = 1024, MANAGE_ITEMS = 4;

__global__ void __launch_bounds__(MANAGE_THREADS)
winner_count_kernel(const int* __restrict__ slot_of, uint64_t num_keys, const uint32_t* __restrict__ keys, unsigned n, unsigned* __restrict__ won)
{
    const unsigned i = blockIdx.x * MANAGE_THREADS + threadIdx.x;
    const uint32_t k = i < n ? keys[i] : NUPS_INVALID_KEY;
    const int all = __syncthreads_count(k < num_keys && slot_of[k] == -(int)(i + 2));
    if (threadIdx.x == 0) won[blockIdx.x] = (unsigned)all;
}

__global__ void __launch_bounds__(MANAGE_THREADS)
assign_counted_kernel(int* slot_of, uint32_t* hot_bits, uint32_t* hot_keys, uint64_t num_keys, const uint32_t* __restrict__ keys,
                      unsigned n, uint64_t H_old, const unsigned* __restrict__ won, unsigned long long* total_out)
{
    __shared__ unsigned before, warp_sum[MANAGE_THREADS / 32];
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * MANAGE_THREADS + threadIdx.x;
    if (threadIdx.x == 0) before = 0;
    __syncthreads();
    unsigned x = threadIdx.x < blockIdx.x ? won[threadIdx.x] : 0u;      // at most as many blocks as threads
    x = __reduce_add_sync(0xFFFFFFFFu, x);
    if (lane == 0 && x) atomicAdd(&before, x);
    const uint32_t k = i < n ? keys[i] : NUPS_INVALID_KEY;
    const bool mine = k < num_keys && slot_of[k] == -(int)(i + 2);
    const unsigned m = __ballot_sync(0xFFFFFFFFu, mine);
    if (lane == 0) warp_sum[warp] = __popc(m);
    __syncthreads();
    unsigned at = before + __popc(m & ((1u << lane) - 1u));
    for (unsigned w = 0; w < warp; ++w) at += warp_sum[w];
    if (mine) {
        slot_of[k] = (int)(H_old + at);
        hot_keys[H_old + at] = k;
        atomicOr(&hot_bits[k >> 5], 1u << (k & 31));
    }
    if (threadIdx.x == 0 && blockIdx.x == gridDim.x - 1) *total_out = before + won[blockIdx.x];
}

// Positions of the flagged items of a round, in order: thread t holds items t * MANAGE_ITEMS ...; returns the position of
// its first one and, in *total, the number of all.  Called by the whole block.
__device__ __forceinline__ unsigned round_positions(const bool (&flag)[MANAGE_ITEMS], unsigned* total)
{
    __shared__ unsigned warp_sum[MANAGE_THREADS / 32];
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned mine = 0;
#pragma unroll
    for (int m = 0; m < (int)MANAGE_ITEMS; ++m) mine += flag[m];
    unsigned inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= (unsigned)o) inc += y;
    }
    __syncthreads();                                         // the round before's readers are done
    if (lane == 31) warp_sum[warp] = inc;
    __syncthreads();
    unsigned before = 0, all = 0;
    for (unsigned w = 0; w < MANAGE_THREADS / 32; ++w) { before += w < warp ? warp_sum[w] : 0u; all += warp_sum[w]; }
    *total = all;
    return before + inc - mine;
}

__global__ void __launch_bounds__(MANAGE_THREADS)
renumber_small_kernel(int* slot_of, uint32_t* hot_keys, unsigned H, unsigned long long* total_out)
{
    unsigned kept = 0;
    for (unsigned b = 0; b < H; b += MANAGE_THREADS * MANAGE_ITEMS) {
        const unsigned first = b + threadIdx.x * MANAGE_ITEMS;
        uint32_t k[MANAGE_ITEMS];
        bool alive[MANAGE_ITEMS];
#pragma unroll
        for (int m = 0; m < (int)MANAGE_ITEMS; ++m) k[m] = first + m < H ? hot_keys[first + m] : 0u;
#pragma unroll
        for (int m = 0; m < (int)MANAGE_ITEMS; ++m) alive[m] = first + m < H && slot_of[k[m]] >= 0;
        unsigned total, at = kept + round_positions(alive, &total);
#pragma unroll
        for (int m = 0; m < (int)MANAGE_ITEMS; ++m) {
            if (!alive[m]) continue;
            slot_of[k[m]] = (int)at;
            hot_keys[at++] = k[m];
        }
        kept += total;
    }
    if (threadIdx.x == 0) *total_out = kept;
}

static nups_status grow_hot(nups_store* s, uint64_t need)
{
    if (need <= s->Hcap) return NUPS_OK;
    uint64_t cap = need + need / 4 + 16;
    uint32_t* hk = nullptr;
    uint32_t* dirty = nullptr;
    float *dv = nullptr, *da = nullptr;
    const size_t slab = (size_t)s->R * cap * s->L * sizeof(float);
    const size_t slab_old = (size_t)s->R * s->Hcap * s->L * sizeof(float);
    const size_t want = cap * 4 + (size_t)s->R * cap * 4 + slab * (s->acc ? 2 : 1);
    const size_t held = s->Hcap * 4 + (size_t)s->R * s->Hcap * 4 + slab_old * (s->acc ? 2 : 1);
    // old and new replicas exist side by side for a moment; the store's limit is judged on what stays
    if (s->dev_cap && (want > s->dev_cap || s->dev_bytes - held > s->dev_cap - want)) return NUPS_ENOMEM;
    const size_t cap_saved = s->dev_cap;
    s->dev_cap = 0;
    bool ok = nups_dev_alloc(s, (void**)&hk, cap * 4) == NUPS_OK &&
              nups_dev_alloc(s, (void**)&dirty, (size_t)s->R * cap * 4) == NUPS_OK &&
              nups_dev_alloc(s, (void**)&dv, slab) == NUPS_OK && (!s->acc || nups_dev_alloc(s, (void**)&da, slab) == NUPS_OK);
    s->dev_cap = cap_saved;
    if (!ok) {
        nups_dev_free(s, hk, cap * 4); nups_dev_free(s, dirty, (size_t)s->R * cap * 4);
        nups_dev_free(s, dv, slab); nups_dev_free(s, da, slab);
        return NUPS_ENOMEM;
    }
    // pending updates are all zero here (the caller merged them), so fresh zeroed slabs are enough
    if (s->H) CK(cudaMemcpy(hk, s->hot_keys, s->H * 4, cudaMemcpyDeviceToDevice));
    CK(cudaMemset(dirty, 0, (size_t)s->R * cap * 4));
    CK(cudaMemset(dv, 0, slab));
    if (da) CK(cudaMemset(da, 0, slab));
    CK(cudaDeviceSynchronize());
    nups_dev_free(s, s->hot_keys, s->Hcap * 4); nups_dev_free(s, s->dirty, (size_t)s->R * s->Hcap * 4);
    nups_dev_free(s, s->dval, slab_old); nups_dev_free(s, s->dacc, slab_old);
    s->hot_keys = hk; s->dirty = dirty; s->dval = dv; s->dacc = da; s->Hcap = cap;
    return NUPS_OK;
}

// The stream is waited for once, at the latest when the call returns, whatever way it returns: the caller may hand the key list
// on, or look at the store from another stream.
static nups_status return_waited(cudaStream_t st, nups_status rc)
{
    CK(cudaStreamSynchronize(st));
    return rc;
}

extern "C" nups_status nups_set_management(nups_store* s, const uint32_t* d_keys, uint64_t n, int technique, void* stream)
{
    if (!s || (n && !d_keys) || (technique != NUPS_SINGLE && technique != NUPS_REPLICATE)) return NUPS_EINVAL;
    if (n >= (1ull << 31) - 2) return NUPS_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    nups_status rc = nups_sync_internal(s, st);
    if (rc != NUPS_OK) return rc;
    if (n == 0) return return_waited(st, NUPS_OK);
    // no background merge may be enqueued or running while slots and replicas are rebuilt
    struct Bracket {
        nups_store* s;
        cudaStream_t st;
        Bracket(nups_store* s_, cudaStream_t st_) : s(s_), st(st_) { nups_background_begin(s, st); }
        ~Bracket() { nups_background_end(s, st); }
    } bracket(s, st);
    uint64_t m = technique == NUPS_REPLICATE ? n : (s->H > n ? s->H : n);
    size_t need = 2 * align256(m * 8) + align256(m * 4) + nups_scan_scratch_bytes(m) + 256;
    char* sc;
    rc = nups_scratch(s, need, &sc);
    if (rc != NUPS_OK) return return_waited(st, rc);
    unsigned long long* flag = (unsigned long long*)sc; sc += align256(m * 8);
    unsigned long long* pos = (unsigned long long*)sc; sc += align256(m * 8);
    uint32_t* hk_new = (uint32_t*)sc; sc += align256(m * 4);
    unsigned long long* d_total = (unsigned long long*)sc; sc += 256;
    unsigned long long total = 0;
    if (technique == NUPS_REPLICATE) {
        if (s->H + n >= (1ull << 31)) return return_waited(st, NUPS_ENOMEM);
        if (s->H + n > s->Hcap) CK(cudaStreamSynchronize(st));           // the merge is done before the replicas move
        rc = grow_hot(s, s->H + n);
        if (rc != NUPS_OK) return rc;
        claim_kernel<<<grid_for(n, 256), 256, 0, st>>>(s->slot_of, s->num_keys, d_keys, n, s->st);
        LAUNCH_CHECK(s);
        if (n <= ASSIGN_LIST_KEYS) {
            unsigned* won = (unsigned*)flag;
            const unsigned blocks = grid_for(n, MANAGE_THREADS);
            winner_count_kernel<<<blocks, MANAGE_THREADS, 0, st>>>(s->slot_of, s->num_keys, d_keys, (unsigned)n, won);
            LAUNCH_CHECK(s);
            assign_counted_kernel<<<blocks, MANAGE_THREADS, 0, st>>>(s->slot_of, s->hot_bits, s->hot_keys, s->num_keys, d_keys, (unsigned)n, s->H, won, d_total);
            LAUNCH_CHECK(s);
        } else {
            winner_flag_kernel<<<grid_for(n, 256), 256, 0, st>>>(s->slot_of, s->num_keys, d_keys, n, flag);
            LAUNCH_CHECK(s);
            rc = nups_scan_u64(s, flag, pos, n, d_total, sc, st);
            if (rc != NUPS_OK) return rc;
            assign_slots_kernel<<<grid_for(n, 256), 256, 0, st>>>(s->slot_of, s->hot_bits, s->hot_keys, d_keys, n, flag, pos, s->H);
            LAUNCH_CHECK(s);
        }
        CK(cudaMemcpyAsync(&total, d_total, 8, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        s->H += total;
    } else {
        demote_kernel<<<grid_for(n, 256), 256, 0, st>>>(s->slot_of, s->hot_bits, s->num_keys, d_keys, n, s->st);
        LAUNCH_CHECK(s);
        if (s->H == 0) return return_waited(st, NUPS_OK);
        if (s->H <= SMALL_LIST_KEYS) {
            renumber_small_kernel<<<1, MANAGE_THREADS, 0, st>>>(s->slot_of, s->hot_keys, (unsigned)s->H, d_total);
            LAUNCH_CHECK(s);
            CK(cudaMemcpyAsync(&total, d_total, 8, cudaMemcpyDeviceToHost, st));
            CK(cudaStreamSynchronize(st));
            s->H = total;
            return NUPS_OK;
        }
        alive_flag_kernel<<<grid_for(s->H, 256), 256, 0, st>>>(s->slot_of, s->hot_keys, s->H, flag);
        LAUNCH_CHECK(s);
        rc = nups_scan_u64(s, flag, pos, s->H, d_total, sc, st);
        if (rc != NUPS_OK) return rc;
        renumber_kernel<<<grid_for(s->H, 256), 256, 0, st>>>(s->slot_of, s->hot_keys, hk_new, s->H, flag, pos);
        LAUNCH_CHECK(s);
        CK(cudaMemcpyAsync(&total, d_total, 8, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        if (total) CK(cudaMemcpyAsync(s->hot_keys, hk_new, total * 4, cudaMemcpyDeviceToDevice, st));
        CK(cudaStreamSynchronize(st));
        s->H = total;
    }
    return NUPS_OK;
}

extern "C" nups_status nups_get_hot(nups_store* s, uint64_t* h_n_out, uint32_t* d_keys_out, void* stream)
{
    if (!s || !h_n_out) return NUPS_EINVAL;
    *h_n_out = s->H;
    if (d_keys_out && s->H) {
        CK(cudaMemcpyAsync(d_keys_out, s->hot_keys, s->H * 4, cudaMemcpyDeviceToDevice, (cudaStream_t)stream));
        CK(cudaStreamSynchronize((cudaStream_t)stream));
    }
    return NUPS_OK;
}

// ---------------------------------------------------------------------------------------------
// ownership (the one-machine reading of "allocated at node q")
// ---------------------------------------------------------------------------------------------
__global__ void localize_request_kernel(View v, const uint32_t* __restrict__ keys, uint64_t n)
{
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t k = keys[i];
    if (k >= v.num_keys) { flag_bad_key(v); return; }
    mark_localize(v, k, worker_of_item(i, n, v.R));
}

extern "C" nups_status nups_localize(nups_store* s, const uint32_t* d_keys, uint64_t n, void* stream)
{
    if (!s || (n && !d_keys) || n >= (1ull << 32)) return NUPS_EINVAL;
    if (!s->own || n == 0) return NUPS_OK;
    cudaStream_t st = (cudaStream_t)stream;
    nups_status rc = nups_new_epoch(s, st);
    if (rc != NUPS_OK) return rc;
    localize_request_kernel<<<grid_for(n, 256), 256, 0, st>>>(nups_view(s), d_keys, n);
    LAUNCH_CHECK(s);
    return NUPS_OK;
}

__global__ void owner_kernel(View v, const uint32_t* __restrict__ keys, uint64_t n, int* __restrict__ out)
{
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t k = keys[i];
    int r;
    if (k >= v.num_keys) r = -1;
    else if (key_is_hot(v, k)) r = -2;
    else if (!v.own) r = -3;
    else r = (v.own[k] & 0xFFu) == NUPS_OWNER_DEFAULT ? (int)(k % v.R) : (int)(v.own[k] & 0xFFu);
    out[i] = r;
}

extern "C" nups_status nups_get_owner(nups_store* s, const uint32_t* d_keys, uint64_t n, int32_t* d_out, void* stream)
{
    if (!s || (n && (!d_keys || !d_out))) return NUPS_EINVAL;
    if (n == 0) return NUPS_OK;
    owner_kernel<<<grid_for(n, 256), 256, 0, (cudaStream_t)stream>>>(nups_view(s), d_keys, n, d_out);
    LAUNCH_CHECK(s);
    return NUPS_OK;
}

// ---------------------------------------------------------------------------------------------
// reduction-rate probe
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
red_probe_kernel(float* base, uint64_t n4)
{
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (; i < n4; i += stride) red_add_v4(base + 4 * i, zero);
}

extern "C" nups_status nups_probe_reduction_rate(nups_store* s, uint64_t bytes, uint32_t reps, double* h_gbs_out, void* stream)
{
    if (!s || !h_gbs_out || reps == 0) return NUPS_EINVAL;
    if (s->vb != 4) return NUPS_ESTATE;                       // the probe adds single-precision zeros
    cudaStream_t st = (cudaStream_t)stream;
    const uint64_t table_bytes = (uint64_t)s->num_keys * s->L * sizeof(float);
    if (bytes > table_bytes) bytes = table_bytes;
    const uint64_t n4 = bytes / 16;
    if (n4 == 0) return NUPS_EINVAL;
    cudaEvent_t a, b;
    CK(cudaEventCreate(&a));
    CK(cudaEventCreate(&b));
    const unsigned grid = grid_for(n4, 256, (unsigned)s->sm_count * 8);
    red_probe_kernel<<<grid, 256, 0, st>>>(s->val, n4);          // warm-up
    CK(cudaEventRecord(a, st));
    for (uint32_t r = 0; r < reps; ++r) red_probe_kernel<<<grid, 256, 0, st>>>(s->val, n4);
    CK(cudaEventRecord(b, st));
    s->launches += reps + 1;
    CK(cudaEventSynchronize(b));
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, a, b));
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    *h_gbs_out = (double)n4 * 16.0 * reps / (ms * 1e-3) / 1e9;
    return NUPS_OK;
}

// ---------------------------------------------------------------------------------------------
// status and statistics
// ---------------------------------------------------------------------------------------------
extern "C" nups_status nups_status_check(nups_store* s, void* stream)
{
    if (!s) return NUPS_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int code = 0;
    CK(cudaMemcpyAsync(&code, &s->st->status, sizeof(int), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (code != 0) {
        CK(cudaMemsetAsync(&s->st->status, 0, sizeof(int), st));
        CK(cudaStreamSynchronize(st));
    }
    return (nups_status)code;
}

extern "C" nups_status nups_get_stats(nups_store* s, uint64_t* h_out, void* stream)
{
    if (!s || !h_out) return NUPS_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    DevStat d;
    CK(cudaMemcpyAsync(&d, s->st, sizeof(DevStat), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    h_out[0] = s->steps; h_out[1] = s->syncs; h_out[2] = s->launches;
    h_out[3] = d.hot_hits; h_out[4] = d.cold_hits; h_out[5] = s->H; h_out[6] = nups_background_merges(s); h_out[7] = 0;
    return NUPS_OK;
}

// Sampling access: register_distribution (alias table built on the device), PrepareSample and
// PullSample under the four conformity levels.  NuPS Sections 4.3, 4.4.
#include <string.h>

#include "nups_internal.cuh"

static inline size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// ---------------------------------------------------------------------------------------------
// Alias table.  n buckets of capacity W = sum w; item j has mass n*w[j]; "lights" have mass < W.
// Lights are topped up by the heavies in index order, and a heavy whose remainder drops below W
// is itself topped up by the next heavy.  With D(a) the running sum of the lights' deficits and
// S(h) the running sum of the heavies' surpluses (both in index order):
//   light a is filled by the first heavy h with S(h) >= D(a-1);
//   heavy h turns light right after the first light a with D(a) > S(h); it keeps
//   W + S(h) - D(a) and is filled by heavy h+1; a heavy that never turns light keeps W.
// ---------------------------------------------------------------------------------------------
__global__ void weight_sum_kernel(const uint32_t* __restrict__ w, uint64_t n, DevStat* st)
{
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    unsigned long long sum = 0;
    for (; i < n; i += stride) sum += w[i];
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(&st->tmp[0], sum);
}

__global__ void alias_classify_kernel(const uint32_t* __restrict__ w, uint64_t n, unsigned long long W,
                                      unsigned long long* __restrict__ lflag, unsigned long long* __restrict__ dfl,
                                      unsigned long long* __restrict__ sfl)
{
    uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    unsigned long long mass = n * (unsigned long long)w[j];
    bool light = mass < W;
    lflag[j] = light ? 1ull : 0ull;
    dfl[j] = light ? W - mass : 0ull;
    sfl[j] = light ? 0ull : mass - W;
}

__global__ void alias_rank_kernel(const uint32_t* __restrict__ w, uint64_t n, unsigned long long W,
                                  const unsigned long long* __restrict__ lrank, const unsigned long long* __restrict__ dex,
                                  const unsigned long long* __restrict__ sex, unsigned long long nL,
                                  unsigned long long* __restrict__ inc /* D at [0,nL), S at [nL,n) */,
                                  uint32_t* __restrict__ hidx)
{
    uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    unsigned long long mass = n * (unsigned long long)w[j];
    unsigned long long a = lrank[j];
    if (mass < W) inc[a] = dex[j] + (W - mass);
    else {
        unsigned long long h = j - a;
        inc[nL + h] = sex[j] + (mass - W);
        hidx[h] = (uint32_t)j;
    }
}

__global__ void alias_fill_kernel(const uint32_t* __restrict__ w, uint64_t n, unsigned long long W,
                                  const unsigned long long* __restrict__ lrank, const unsigned long long* __restrict__ dex,
                                  unsigned long long nL, const unsigned long long* __restrict__ inc,
                                  const uint32_t* __restrict__ hidx, AliasEntry* __restrict__ table)
{
    uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const unsigned long long* D = inc;
    const unsigned long long* S = inc + nL;
    const unsigned long long nH = n - nL;
    unsigned long long mass = n * (unsigned long long)w[j];
    AliasEntry e;
    e.pad = 0;
    if (mass < W) {
        unsigned long long target = dex[j];          // D(a-1)
        unsigned long long lo = 0, hi = nH;          // first h with S[h] >= target
        while (lo < hi) {
            unsigned long long mid = (lo + hi) >> 1;
            if (S[mid] >= target) hi = mid; else lo = mid + 1;
        }
        e.thr = mass;
        e.alias = hidx[lo < nH ? lo : nH - 1];
    } else {
        unsigned long long h = j - lrank[j];
        unsigned long long Sh = S[h];
        unsigned long long lo = 0, hi = nL;          // first a with D[a] > Sh
        while (lo < hi) {
            unsigned long long mid = (lo + hi) >> 1;
            if (D[mid] > Sh) hi = mid; else lo = mid + 1;
        }
        if (lo < nL && h + 1 < nH) {
            e.thr = W + Sh - D[lo];
            e.alias = hidx[h + 1];
        } else {
            e.thr = W;
            e.alias = (uint32_t)j;
        }
    }
    table[j] = e;
}

__global__ void alias_unpack_kernel(const AliasEntry* __restrict__ table, uint64_t n, unsigned long long* thr,
                                    uint32_t* alias)
{
    uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    thr[j] = table[j].thr;
    alias[j] = table[j].alias;
}

extern "C" nups_status nups_register_distribution(nups_store* s, uint32_t key_base, const uint32_t* d_weights,
                                                  uint64_t n, int level, uint32_t U, uint32_t G, uint64_t seed,
                                                  int32_t* h_dist_out, void* stream)
{
    if (!s || !h_dist_out) return NUPS_EINVAL;
    if (n == 0 || (uint64_t)key_base + n > s->num_keys) return NUPS_EINVAL;
    if (level < NUPS_CONFORM || level > NUPS_NONCONFORM) return NUPS_EINVAL;
    bool reuse = level == NUPS_BOUNDED || level == NUPS_LONGTERM;
    if (reuse && (U == 0 || G == 0 || G > NUPS_MAX_POOL)) return NUPS_EINVAL;
    if ((level == NUPS_LONGTERM || level == NUPS_NONCONFORM) && !s->own) return NUPS_ESTATE;
    int id = -1;
    for (int i = 0; i < NUPS_MAX_DISTS; ++i) if (!s->dist[i].used) { id = i; break; }
    if (id < 0) return NUPS_ENOMEM;
    cudaStream_t st = (cudaStream_t)stream;
    Dist d;
    memset(&d, 0, sizeof(d));
    d.key_base = key_base; d.n = n; d.level = level; d.U = U; d.G = G; d.seed = seed;
    if (!d_weights) d.uniform = 1;
    else {
        CK(cudaMemsetAsync(&s->st->tmp[0], 0, 8, st));
        weight_sum_kernel<<<grid_for(n, 256, (unsigned)s->sm_count * 8), 256, 0, st>>>(d_weights, n, s->st);
        LAUNCH_CHECK(s);
        unsigned long long W = 0;
        CK(cudaMemcpyAsync(&W, &s->st->tmp[0], 8, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        if (W == 0) return NUPS_EINVAL;
        unsigned __int128 nW = (unsigned __int128)W * n;
        if (nW >> 64) return NUPS_EINVAL;
        d.W = W;
        size_t need = 4 * align256(n * 8) + align256(n * 4) + nups_scan_scratch_bytes(n) + 256;
        char* sc;
        nups_status rc = nups_scratch(s, need, &sc);
        if (rc != NUPS_OK) return rc;
        unsigned long long* lrank = (unsigned long long*)sc; sc += align256(n * 8);
        unsigned long long* dex = (unsigned long long*)sc; sc += align256(n * 8);
        unsigned long long* sex = (unsigned long long*)sc; sc += align256(n * 8);
        unsigned long long* inc = (unsigned long long*)sc; sc += align256(n * 8);
        uint32_t* hidx = (uint32_t*)sc; sc += align256(n * 4);
        unsigned long long* d_nL = (unsigned long long*)sc; sc += 256;
        rc = nups_dev_alloc(s, &d.table, n * sizeof(AliasEntry));
        if (rc != NUPS_OK) return rc;
        unsigned g = grid_for(n, 256);
        alias_classify_kernel<<<g, 256, 0, st>>>(d_weights, n, W, lrank, dex, sex);
        LAUNCH_CHECK(s);
        rc = nups_scan_u64(s, lrank, lrank, n, d_nL, sc, st);
        if (rc == NUPS_OK) rc = nups_scan_u64(s, dex, dex, n, nullptr, sc, st);
        if (rc == NUPS_OK) rc = nups_scan_u64(s, sex, sex, n, nullptr, sc, st);
        if (rc != NUPS_OK) { nups_dev_free(s, d.table, n * sizeof(AliasEntry)); return rc; }
        unsigned long long nL = 0;
        CK(cudaMemcpyAsync(&nL, d_nL, 8, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        alias_rank_kernel<<<g, 256, 0, st>>>(d_weights, n, W, lrank, dex, sex, nL, inc, hidx);
        LAUNCH_CHECK(s);
        alias_fill_kernel<<<g, 256, 0, st>>>(d_weights, n, W, lrank, dex, nL, inc, hidx, (AliasEntry*)d.table);
        LAUNCH_CHECK(s);
        CK(cudaStreamSynchronize(st));
    }
    if (nups_dev_alloc(s, (void**)&d.off, 2 * s->R * 8) != NUPS_OK) {
        nups_dev_free(s, d.table, d.table ? n * sizeof(AliasEntry) : 0);
        return NUPS_ENOMEM;
    }
    CK(cudaMemsetAsync(d.off, 0, 2 * s->R * 8, st));
    CK(cudaStreamSynchronize(st));
    d.used = 1;
    s->dist[id] = d;
    *h_dist_out = id;
    return NUPS_OK;
}

extern "C" nups_status nups_get_alias_table(nups_store* s, int32_t dist, uint64_t* d_thr_out, uint32_t* d_alias_out,
                                            uint64_t* h_W_out, void* stream)
{
    if (!s || dist < 0 || dist >= NUPS_MAX_DISTS || !s->dist[dist].used) return NUPS_EINVAL;
    Dist& d = s->dist[dist];
    if (h_W_out) *h_W_out = d.W;
    if (d.uniform) return d_thr_out || d_alias_out ? NUPS_EINVAL : NUPS_OK;
    if (d_thr_out && d_alias_out) {
        alias_unpack_kernel<<<grid_for(d.n, 256), 256, 0, (cudaStream_t)stream>>>((const AliasEntry*)d.table, d.n,
                                                                              (unsigned long long*)d_thr_out, d_alias_out);
        LAUNCH_CHECK(s);
    }
    return NUPS_OK;
}

// ---------------------------------------------------------------------------------------------
// Draws
// ---------------------------------------------------------------------------------------------
struct DrawParams {
    const AliasEntry* table;
    unsigned long long n, W, seed;
    uint32_t key_base, U, G;
    int uniform;
};

static DrawParams draw_params(const Dist& d)
{
    DrawParams p;
    p.table = (const AliasEntry*)d.table; p.n = d.n; p.W = d.W; p.seed = d.seed;
    p.key_base = d.key_base; p.U = d.U; p.G = d.G; p.uniform = d.uniform;
    return p;
}

// one iid draw from pi: position `pos` of worker q's stream; 64 bits pick the bucket, 64 bits the
// point inside it.  In two halves, so that the bucket's table entry can be on its way while other work is done.
struct Draw {
    unsigned long long j, b;
    AliasEntry e;
};
__device__ __forceinline__ Draw draw_begin(const DrawParams& p, uint32_t q, unsigned long long pos)
{
    uint32_t x[4];
    philox_at(p.seed, pos, q, 0, 0, x);
    const unsigned long long a = (unsigned long long)x[0] | ((unsigned long long)x[1] << 32);
    Draw d;
    d.b = (unsigned long long)x[2] | ((unsigned long long)x[3] << 32);
    d.j = __umul64hi(a, p.n);
    if (!p.uniform) d.e = p.table[d.j];
    return d;
}
__device__ __forceinline__ uint32_t draw_end(const DrawParams& p, const Draw& d)
{
    const bool own = p.uniform || __umul64hi(d.b, p.W) < d.e.thr;
    return p.key_base + (own ? (uint32_t)d.j : d.e.alias);
}
__device__ __forceinline__ uint32_t draw_iid(const DrawParams& p, uint32_t q, unsigned long long pos)
{
    return draw_end(p, draw_begin(p, q, pos));
}

// Handle buffer layout (device): keys[N] (u32) | post[N] (u32) | state[3][R] (uint4) | flags | prefix
struct HandleView {
    uint32_t* keys;
    uint32_t* post;    // LONG-TERM: postponed entries of each sub-handle, in the order they were postponed
    uint4* state;      // LONG-TERM per sub-handle: x = walk position, y = postponed head, z = postponed tail
    uint4* prev;       //   the state before the running call
    uint4* walk;       //   what the running call does: x = fresh entries walked, y = of those local,
                       //   z = postponed entries emitted, w = blocks that have looked up their part (0 between calls)
    uint32_t* flags;   // LONG-TERM: "is local" bit of every fresh entry, and the number of local entries before
    uint32_t* prefix;  //   each 32-entry word; sub-handle q owns the words from (b_q / 32) + q on
};
static size_t handle_bytes(uint64_t N, uint32_t R, int level)
{
    size_t b = align256(N * 4);
    if (level == NUPS_LONGTERM) b += align256(N * 4) + 3 * align256((size_t)R * 16) + 2 * align256((N / 32 + R + 2) * 4);
    return b;
}
static HandleView handle_view(char* buf, uint64_t N, uint32_t R, int level)
{
    HandleView h;
    memset(&h, 0, sizeof(h));
    h.keys = (uint32_t*)buf; buf += align256(N * 4);
    if (level == NUPS_LONGTERM) {
        h.post = (uint32_t*)buf; buf += align256(N * 4);
        h.state = (uint4*)buf; buf += align256((size_t)R * 16);
        h.prev = (uint4*)buf; buf += align256((size_t)R * 16);
        h.walk = (uint4*)buf; buf += align256((size_t)R * 16);
        h.flags = (uint32_t*)buf; buf += align256((N / 32 + R + 2) * 4);
        h.prefix = (uint32_t*)buf; buf += align256((N / 32 + R + 2) * 4);
    }
    return h;
}

// Local sampling: the first key local to worker q among the candidate k0 and the 63 keys after it
// (wrapping inside the distribution's key range), else k0.  The candidates are consecutive keys, so
// their ownership words are consecutive too.  Four lanes serve one candidate: each reads the four words
// of its part of a 16-key group with one 128-bit load (the four loads of a candidate fall into one cache
// line, so a warp instruction touches 8 lines instead of 32), and the walk goes group by group until
// a local key shows up (most walks end within the first group).
// Called by all four lanes of a quad with the same arguments; whole warps must call.
__device__ __forceinline__ uint32_t first_local_quad(const View& v, const DrawParams& p, uint32_t q, uint32_t k0,
                                                     bool active)
{
    const unsigned sub = threadIdx.x & 3;
    const uint32_t R = v.R;
    uint32_t result = k0;
    bool searching = active && v.own != nullptr;
    const unsigned long long rel = k0 - p.key_base;
    const uint32_t a0 = k0 & ~3u;                            // 16-byte aligned start
    if (searching && !(rel + NUPS_LOCAL_PROBES <= p.n && (uint64_t)a0 + NUPS_LOCAL_PROBES + 16 <= v.num_keys)) {
        // near the end of the key range: probe one key at a time
        for (uint32_t probe = 0; probe < NUPS_LOCAL_PROBES; ++probe) {
            const uint32_t cand = p.key_base + (uint32_t)((rel + probe) % p.n);
            if (key_is_local(v, q, cand)) { result = cand; break; }
        }
        searching = false;
    }
    const uint32_t res0 = searching ? a0 % R : 0u;           // key mod R of key a0
    for (uint32_t g = 0; g < NUPS_LOCAL_PROBES / 16 + 1; ++g) {
        if (!__any_sync(0xFFFFFFFFu, searching)) break;
        uint32_t m = 0;                                      // bit t: my key t is a candidate and local
        const uint32_t kb = a0 + 16 * g + 4 * sub;           // my four keys: kb ... kb + 3
        if (searching) {
            const uint4 o = __ldg(reinterpret_cast<const uint4*>(v.own + kb));
            const uint32_t hw = v.H ? __ldg(v.hot_bits + (kb >> 5)) >> (kb & 31) : 0u;     // replicated: local to all
            uint32_t r = (res0 + 16 * g + 4 * sub) % R;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const uint32_t w = t == 0 ? o.x : t == 1 ? o.y : t == 2 ? o.z : o.w;
                const uint32_t ob = w & 0xFFu;
                const bool loc = (ob == NUPS_OWNER_DEFAULT ? r : ob) == q || ((hw >> t) & 1u);
                const uint32_t key = kb + t;
                if (loc && key >= k0 && key - k0 < NUPS_LOCAL_PROBES) m |= 1u << t;
                r = r + 1 == R ? 0u : r + 1;
            }
            m <<= 4 * sub;
        }
        m |= __shfl_xor_sync(0xFFFFFFFFu, m, 1);
        m |= __shfl_xor_sync(0xFFFFFFFFu, m, 2);
        if (searching && m) {
            result = a0 + 16 * g + (uint32_t)(__ffs(m) - 1);
            searching = false;
        }
    }
    return result;
}

// one candidate per lane: the quads take the warp's candidates eight at a time
__device__ __forceinline__ uint32_t first_local_warp(const View& v, const DrawParams& p, uint32_t q, uint32_t k0,
                                                     bool active)
{
    const unsigned lane = threadIdx.x & 31;
    uint32_t mine = k0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int src = 8 * r + (int)(lane >> 2);
        const uint32_t kk = __shfl_sync(0xFFFFFFFFu, k0, src);
        const uint32_t qq = __shfl_sync(0xFFFFFFFFu, q, src);
        const bool act = __shfl_sync(0xFFFFFFFFu, (int)active, src) != 0;
        const uint32_t res = first_local_quad(v, p, qq, kk, act);
        const uint32_t back = __shfl_sync(0xFFFFFFFFu, res, 4 * (int)(lane & 7));
        if ((int)(lane >> 3) == r) mine = back;
    }
    return mine;
}

// independent draws: one thread per sample.  The advanced stream offsets go to the other half of the
// distribution's offset array.
__global__ void draw_iid_kernel(View v, DrawParams p, const unsigned long long* __restrict__ off_cur,
                                unsigned long long* __restrict__ off_next, HandleView h, uint64_t N, int localize)
{
    grid_dependency_wait();
    const uint32_t R = v.R;
    if (blockIdx.x == 0)
        for (uint32_t w = threadIdx.x; w < R; w += blockDim.x)
            off_next[w] = off_cur[w] + (chunk_begin(w + 1, N, R) - chunk_begin(w, N, R));
    uint64_t o = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= N) return;
    const uint32_t q = chunk_of_pos(o, N, R);
    const uint32_t k = draw_iid(p, q, off_cur[q] + (o - chunk_begin(q, N, R)));
    h.keys[o] = k;
    if (localize)                                  // PrepareSample localizes what it sampled
        mark_localize_rare(v, k, q, __popc(__match_any_sync(__activemask(), k)) > 1);
}

// Pooled reuse: pool `pl` of a worker holds G iid draws and is walked U times, each pass in a fresh
// Fisher-Yates order.  Stream position s lies in pass number s / G overall (pool = pass / U).
// One block visits one pool, one warp makes one pass at a time, only the passes that are asked for.
// A shuffle swaps positions i and r_i for i = G-1 ... 1 (r_i <= i, drawn beforehand), a chain of dependent swaps.  All that
// depends on their order is who wrote a position last: position i is final after step i, and holds what position r_i held
// before it, which is what position j held before step j if j > i was the last step to write there (r_j = r_i), and r_i
// itself if none was; and likewise for position j.  So the warp takes 32 steps at once and notes for each the last step
// before it that wrote position r_i: one of the 32, found by comparing the r_i bit by bit with ballots, or what the steps
// before left in last[r_i].  All positions then follow these notes side by side.  (The longest chain of notes of a shuffle
// has no bound below G; over 2,000 shuffles of 250 positions it was 6.6 on average and 14 at most, of 1,024 positions 8.7 and 15.)
// Measured, pools of 250 with 16 passes: 19 -> 14 us for 1M samples, 16 -> 10 us for sixteen batches of 12,288, where one thread
// per pass made the swaps (11,000 of 22,000 cycles; noting the steps one by one still takes 8,500).
// Shared memory: pool[G] (u32) | step[T][P] (u16) | last[T][P] (u16).
constexpr unsigned REUSE_THREADS = 512;
struct ReuseShape {
    unsigned T;
    size_t smem;
};
__host__ __device__ inline uint32_t reuse_pitch(uint32_t G) { return (G + 1) / 2 * 2; }     // arrays of whole 32-bit words
static ReuseShape reuse_shape(uint32_t U, uint32_t G)
{
    const size_t pass = (size_t)reuse_pitch(G) * 4;
    ReuseShape r;
    r.T = U < REUSE_THREADS / 32 ? U : REUSE_THREADS / 32;
    while (r.T > 1 && r.T * pass > 40 * 1024) r.T--;
    r.smem = (size_t)G * 4 + r.T * pass;
    return r;
}
static unsigned reuse_pools(uint64_t max_size, uint32_t U, uint32_t G)
{
    return (unsigned)(max_size / ((uint64_t)U * G) + 2);      // a stretch may begin and end inside a pool
}

// emit(in, key, position in the stretch, mark): called by whole warps for every output position; `mark` says
// whether the key still has to be localized there.  When a whole pass of the pool lies inside the stretch, every
// key of the pool is sampled by this call, so the pool's keys are localized once each (mark_key) instead of once
// per output position (U times as often).
template <class Emit, class Mark>
__device__ __forceinline__ void reuse_pool_visit(const DrawParams& p, uint32_t q, unsigned long long s0,
                                                 unsigned long long s1, uint32_t T, Emit emit, Mark mark_key)
{
    extern __shared__ __align__(16) uint32_t reuse_mem[];
    constexpr uint32_t NONE = 0xFFFFu, FIRST = 0x8000u, DRAWS = (NUPS_MAX_POOL + REUSE_THREADS - 1) / REUSE_THREADS;
    constexpr unsigned FULL = 0xFFFFFFFFu;
    static_assert(NUPS_MAX_POOL < FIRST, "a position of a pool and one mark fit 16 bits");
    const uint32_t G = p.G, U = p.U, P = reuse_pitch(G);
    const unsigned tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned long long span = (unsigned long long)U * G;
    const unsigned long long pl = s0 / span + blockIdx.x;
    if (pl * span >= s1) return;
    uint32_t* pool = reuse_mem;
    // passes of this pool that overlap the stretch; does one of them lie fully inside?
    const unsigned long long pool_first = pl * U, pool_end = pool_first + U, lo = s0 / G, hi = (s1 + G - 1) / G;
    const unsigned long long pass_first = lo > pool_first ? lo : pool_first, pass_end = hi < pool_end ? hi : pool_end;
    const unsigned long long whole_first = (s0 + G - 1) / G, whole_end = s1 / G;
    const bool whole_pass = (whole_first > pool_first ? whole_first : pool_first) < (whole_end < pool_end ? whole_end : pool_end);
    Draw drawn[DRAWS];                                       // the pool's keys, on their way while the first shuffles are made
#pragma unroll
    for (unsigned m = 0; m < DRAWS; ++m)
        if (tid + m * REUSE_THREADS < G) drawn[m] = draw_begin(p, q, pl * G + tid + m * REUSE_THREADS);
    const uint32_t blocks_per_pass = (G + 2) / 4;            // Philox blocks that hold the G - 1 shuffle words
    const unsigned bits = 32 - __clz((int)(G - 1) | 1);      // of a position
    uint16_t* st = reinterpret_cast<uint16_t*>(reuse_mem + G) + warp * P;          // this warp's pass (warps below T)
    uint16_t* la = reinterpret_cast<uint16_t*>(reuse_mem + G) + (size_t)T * P + warp * P;
    bool drawing = true;
    for (unsigned long long pass0 = pass_first; pass0 < pass_end; pass0 += T) {
        const unsigned long long pass = pass0 + warp;
        const bool mine = warp < T && pass < pass_end;
        if (mine) {
            __syncwarp();                                    // the pass before is handed out
            // swap partners: step i = G-1 ... 1 of a pass swaps i with mulhi(x, i + 1), x = word G-1-i of the
            // pass's Philox stream (purpose 1, four words per block)
            for (uint32_t blk = lane; blk < blocks_per_pass; blk += 32) {
                uint32_t x[4];
                philox_at(p.seed, pass, q, 1, blk, x);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t d = blk * 4 + k;
                    if (d + 1 < G) st[G - 1 - d] = (uint16_t)__umulhi(x[k], G - d);
                }
            }
            if (lane == 0) st[0] = 0;
            for (uint32_t e = lane; e < P; e += 32) la[e] = (uint16_t)NONE;
            __syncwarp();
            for (int top = (int)G - 1; top >= 0; top -= 32) {            // steps top, top - 1, ...: lane 0 comes first
                const int i = top - (int)lane;
                const uint32_t r = i >= 0 ? st[i] : 0u;
                const unsigned writers = __ballot_sync(FULL, i >= 0 && r != (uint32_t)i);       // others swap with themselves
                unsigned same = writers;
                for (unsigned bit = 0; bit < bits; ++bit) {
                    const unsigned ones = __ballot_sync(FULL, (r >> bit) & 1u);
                    same &= (r >> bit) & 1u ? ones : ~ones;
                }
                const unsigned earlier = same & ((1u << lane) - 1u), later = same & ~((2u << lane) - 1u);
                const uint32_t left = la[r];
                __syncwarp();
                if (i >= 0) {
                    if ((writers >> lane & 1u) && !later) la[r] = (uint16_t)i;
                    const uint32_t before = earlier ? (uint32_t)(top - (31 - __clz((int)earlier))) : left;
                    st[i] = (uint16_t)(before == NONE ? FIRST | r : before);
                }
                __syncwarp();
            }
        }
        if (drawing) {
#pragma unroll
            for (unsigned m = 0; m < DRAWS; ++m) {
                if (tid + m * REUSE_THREADS >= G) continue;
                const uint32_t k = draw_end(p, drawn[m]);
                pool[tid + m * REUSE_THREADS] = k;
                if (whole_pass) mark_key(k);
            }
            __syncthreads();
            drawing = false;
        }
        if (mine) {
            for (uint32_t j0 = 0; j0 < G; j0 += 32) {        // whole warps: emit may ballot
                const uint32_t j = j0 + lane;
                const unsigned long long sp = pass * G + j;
                const bool in = j < G && sp >= s0 && sp < s1;
                uint32_t x = in ? st[j] : FIRST;
                if (x & FIRST) x &= FIRST - 1;
                else
                    for (uint32_t y; (y = la[x]) != NONE;) x = y;
                emit(in, in ? pool[x] : 0u, sp - s0, !whole_pass);
            }
        }
    }
}

__global__ void draw_reuse_kernel(View v, DrawParams p, const unsigned long long* __restrict__ off_cur,
                                  unsigned long long* __restrict__ off_next, HandleView h, uint64_t N, int localize,
                                  int longterm, uint32_t T)
{
    grid_dependency_wait();
    const uint32_t q = blockIdx.y, R = v.R;
    const unsigned long long b0 = chunk_begin(q, N, R), size = chunk_begin(q + 1, N, R) - b0;
    const unsigned long long s0 = off_cur[q];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        off_next[q] = s0 + size;
        if (longterm) h.state[q] = h.walk[q] = make_uint4(0u, 0u, 0u, 0u);
    }
    if (size == 0) return;
    reuse_pool_visit(p, q, s0, s0 + size, T, [&](bool in, uint32_t k, unsigned long long rel, bool mark) {
        if (in) {
            h.keys[b0 + rel] = k;
            if (localize && mark) mark_localize(v, k, q);
        }
    }, [&](uint32_t k) { if (localize) mark_localize(v, k, q); });
}

static nups_status prepare_internal(nups_store* s, int32_t dist, uint64_t N, int* slot_out, cudaStream_t st)
{
    if (dist < 0 || dist >= NUPS_MAX_DISTS || !s->dist[dist].used || N == 0 || N >= (1ull << 32)) return NUPS_EINVAL;
    if (s->ahead_dist == dist) {
        nups_status rw = nups_sample_ahead_rewind(s, st);       // samples drawn ahead for the steps go back
        if (rw != NUPS_OK) return rw;
    }
    Dist& d = s->dist[dist];
    size_t need = handle_bytes(N, s->R, d.level);
    int id = -1;
    for (int i = 0; i < NUPS_MAX_HANDLES && id < 0; ++i)
        if (!s->handle[i].used && s->handle[i].cap >= need) id = i;      // reuse a released buffer
    for (int i = 0; i < NUPS_MAX_HANDLES && id < 0; ++i)
        if (!s->handle[i].used && s->handle[i].cap == 0) id = i;
    for (int i = 0; i < NUPS_MAX_HANDLES && id < 0; ++i)
        if (!s->handle[i].used) id = i;
    if (id < 0) return NUPS_ENOMEM;
    Handle& h = s->handle[id];
    if (h.cap < need) {
        size_t want = need + need / 4;
        if (s->dev_cap && (want > s->dev_cap || s->dev_bytes - h.cap > s->dev_cap - want)) return NUPS_ENOMEM;
        nups_dev_free(s, h.buf, h.cap);
        h.buf = nullptr; h.cap = 0;
        nups_status rc = nups_dev_alloc(s, (void**)&h.buf, want);
        if (rc != NUPS_OK) return rc;
        h.cap = want;
    }
    const bool reuse = d.level == NUPS_BOUNDED || d.level == NUPS_LONGTERM;
    const bool loc = s->own && d.level != NUPS_NONCONFORM;
    if (loc) {
        nups_status rc = nups_new_epoch(s, st);
        if (rc != NUPS_OK) return rc;
    }
    HandleView hv = handle_view(h.buf, N, s->R, d.level);
    DrawParams p = draw_params(d);
    View v = nups_view(s);
    const unsigned long long* off_cur = d.off + (size_t)d.cur * s->R;
    unsigned long long* off_next = d.off + (size_t)(d.cur ^ 1) * s->R;
    nups_time_begin(s, st, NUPS_TIMED_DRAW);
    if (reuse) {
        const ReuseShape sh = reuse_shape(d.U, d.G);
        nups_launch_dependent(draw_reuse_kernel, dim3(reuse_pools((N + s->R - 1) / s->R, d.U, d.G), s->R), REUSE_THREADS,
                              sh.smem, st, v, p, off_cur, off_next, hv, N, loc, d.level == NUPS_LONGTERM, sh.T);
    } else {
        nups_launch_dependent(draw_iid_kernel, grid_for(N, 256), 256, 0, st, v, p, off_cur, off_next, hv, N, loc);
    }
    nups_time_end(s, st);
    LAUNCH_CHECK(s);
    d.cur ^= 1;
    h.used = 1; h.dist = dist; h.N = N; h.cursor = 0;
    *slot_out = id;
    return NUPS_OK;
}

extern "C" nups_status nups_prepare_sample(nups_store* s, int32_t dist, uint64_t N, nups_handle* h_out, void* stream)
{
    if (!s || !h_out) return NUPS_EINVAL;
    int id = -1;
    nups_status rc = prepare_internal(s, dist, N, &id, (cudaStream_t)stream);
    if (rc == NUPS_OK) *h_out = id;
    return rc;
}

// ---------------------------------------------------------------------------------------------
// PullSample
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void count_sample(const View& v, uint32_t key, bool emitted)
{
    if (!v.count) return;
    const unsigned lane = threadIdx.x & 31;
    bool hot = emitted && key_is_hot(v, key);
    if (emitted) atomicAdd(v.cnt + key, 1ull);
    unsigned hot_m = __ballot_sync(0xFFFFFFFFu, emitted && hot);
    unsigned cold_m = __ballot_sync(0xFFFFFFFFu, emitted && !hot);
    if (lane == 0) {
        if (hot_m) atomicAdd(&v.st->hot_hits, (unsigned long long)__popc(hot_m));
        if (cold_m) atomicAdd(&v.st->cold_hits, (unsigned long long)__popc(cold_m));
    }
}

// independent draws / pooled reuse: the keys were fixed at PrepareSample.
// local sampling: first key local to the worker at or after the candidate.
__global__ void emit_kernel(View v, DrawParams p, HandleView h, uint64_t N, uint64_t cursor, uint64_t n, int local_only,
                            uint32_t* __restrict__ out)
{
    grid_dependency_wait();
    uint64_t o = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool in = o < n;
    uint32_t k = 0;
    uint32_t q = 0;
    if (in) {
        k = h.keys[cursor + o];
        if (local_only) q = chunk_of_pos(cursor + o, N, v.R);
    }
    if (local_only) k = first_local_warp(v, p, q, k, in);
    if (in) out[o] = k;
    count_sample(v, k, in);
}

// Reuse with postponing.  Entries of a sub-handle not yet postponed are taken in list order: a local
// one is emitted, a non-local one is re-localized and appended to the sub-handle's postponed queue;
// the walk stops right after the last entry it must emit, and when the fresh entries run out the
// postponed ones are emitted.  Locality is judged by the ownership at the start of the call.
// Where an entry goes depends only on how many local entries lie before it, so the walk is a
// prefix sum, not a loop: one bit per fresh entry, looked up by the whole GPU; per sub-handle, a scan of the bit
// counts that also finds where the walk stops, made by the block that is the last to have looked up its part; then
// every entry is placed on its own, and what is postponed moves to its worker.
struct LtChunk {
    uint32_t q;
    uint64_t b0, size, take, out_base;
    bool active;
};
__device__ __forceinline__ LtChunk lt_chunk(uint32_t q, uint64_t N, uint32_t R, uint64_t cursor, uint64_t n)
{
    LtChunk c;
    c.q = q;
    c.b0 = chunk_begin(q, N, R);
    const uint64_t b1 = chunk_begin(q + 1, N, R);
    const uint64_t lo = max(c.b0, cursor), hi = min(b1, cursor + n);
    c.active = lo < hi;
    c.size = b1 - c.b0;
    c.take = c.active ? hi - lo : 0;
    c.out_base = c.active ? lo - cursor : 0;
    return c;
}

// Lookups and scan in one launch, as the calls are bound by their launches: drawing 120,000 samples and pulling them in four
// parts 91 -> 74 us with this and the rows copied by the placement pass, 1M samples in one part 134 -> 130 us, in four 186 -> 184 us
// (135 and 193 us with twice as many blocks as are resident).  A block that has written its bits makes them visible and takes
// a ticket; the one that draws the last of its sub-handle's tickets sees all of them and scans.  Nobody waits for anybody.
constexpr int LT_THREADS = 512;
constexpr unsigned LT_BLOCKS = 2;            // resident per multiprocessor
constexpr int LT_WORDS = 4;                  // flag words per thread and round of the scan

__global__ void __launch_bounds__(LT_THREADS, LT_BLOCKS)
lt_walk_kernel(View v, HandleView h, uint64_t N, uint64_t cursor, uint64_t n, uint32_t q_first)
{
    grid_dependency_wait();
    __shared__ unsigned warp_tot[LT_THREADS / 32];
    __shared__ unsigned long long sh_stop;       // walk position right after the last entry that must be emitted
    __shared__ bool sh_last;
    const LtChunk c = lt_chunk(q_first + blockIdx.y, N, v.R, cursor, n);
    if (!c.active) return;
    const unsigned tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint4 stt = h.state[c.q];
    const uint64_t oc = stt.x, ph = stt.y, pt = stt.z;
    const uint64_t w0 = oc >> 5, w1 = oc < c.size ? (c.size + 31) >> 5 : w0;
    uint32_t* flags = h.flags + (c.b0 >> 5) + c.q;
    uint32_t* prefix = h.prefix + (c.b0 >> 5) + c.q;
    {
        const uint64_t stride = (uint64_t)gridDim.x * (LT_THREADS / 32);
        for (uint64_t word = w0 + (uint64_t)blockIdx.x * (LT_THREADS / 32) + warp; word < w1; word += stride) {
            const uint64_t i = word * 32 + lane;
            const bool loc = i >= oc && i < c.size && key_is_local(v, c.q, h.keys[c.b0 + i]);
            const unsigned bits = __ballot_sync(0xFFFFFFFFu, loc);
            if (lane == 0) flags[word] = bits;
        }
    }
    __syncthreads();
    if (tid == 0) {
        // orders the block's bits (the barrier puts them before this) before the ticket, and the ticket before the scan's
        // reads of the other blocks' bits; a fence by every warp that wrote bits took 14 us more for 1M samples
        __threadfence();
        const unsigned ticket = atomicAdd(&h.walk[c.q].w, 1u);
        __threadfence();
        sh_last = ticket == gridDim.x - 1;
        sh_stop = ~0ull;
    }
    __syncthreads();
    if (!sh_last) return;
    unsigned long long carry = 0;                // local entries before the round
    for (uint64_t base = w0; base < w1 && carry < c.take; base += (uint64_t)LT_THREADS * LT_WORDS) {
        uint32_t bits[LT_WORDS];
        unsigned mine = 0;
#pragma unroll
        for (int k = 0; k < LT_WORDS; ++k) {
            const uint64_t w = base + (uint64_t)tid * LT_WORDS + k;
            bits[k] = w < w1 ? __ldcg(flags + w) : 0u;         // written by other multiprocessors
            mine += __popc(bits[k]);
        }
        unsigned inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= (unsigned)o) inc += y;
        }
        if (lane == 31) warp_tot[warp] = inc;
        __syncthreads();
        unsigned long long before = carry + (inc - mine);
        unsigned total = 0;
        for (unsigned w = 0; w < LT_THREADS / 32; ++w) {
            if (w < warp) before += warp_tot[w];
            total += warp_tot[w];
        }
#pragma unroll
        for (int k = 0; k < LT_WORDS; ++k) {
            const uint64_t w = base + (uint64_t)tid * LT_WORDS + k;
            if (w < w1) prefix[w] = (uint32_t)before;
            const unsigned cnt = __popc(bits[k]);
            if (before < c.take && c.take <= before + cnt) {
                // the take-th local entry is the (take - before)-th set bit of this word
                uint32_t b = bits[k];
                for (unsigned long long skip = c.take - before - 1; skip; --skip) b &= b - 1;
                sh_stop = w * 32 + (unsigned)(__ffs(b) - 1) + 1;
            }
            before += cnt;
        }
        carry += total;
        __syncthreads();
    }
    __syncthreads();
    if (tid == 0) {
        const uint64_t fresh = oc < c.size ? c.size - oc : 0;
        const uint64_t tc = carry >= c.take ? (uint64_t)sh_stop - oc : fresh;      // fresh entries walked
        const uint64_t tl = carry >= c.take ? c.take : (uint64_t)carry;             // of those local = emitted
        const uint64_t cnt = c.take - tl;                                           // postponed entries emitted
        h.prev[c.q] = stt;
        h.walk[c.q] = make_uint4((unsigned)tc, (unsigned)tl, (unsigned)cnt, 0u);
        h.state[c.q] = make_uint4((unsigned)(oc + tc), (unsigned)(ph + cnt), (unsigned)(pt + tc - tl), 0u);
    }
}

// C8 > 0: the kernel also copies the rows of the keys it emits (rows of C8 chunks of 32 bytes, 32 / C8 rows per warp
// instruction, as gather8_kernel does), which saves the separate gather launch of a PullSample with values.  The 32 entries
// of a word are then shared by `sharers` warps (1, 2 or 4): all of them find out where the entries go, the first one writes
// that down, and each copies its part of the rows.  A call on two sub-handles of 15,000 entries has 940 words, and one warp
// per word waited for four rows at a time eight times over.  Measured: 21,756 samples of 128 floats in four parts 68.0 -> 50.1 us, 14,380
// of 64 floats in one 21.8 -> 19.5 us.  UNR: instructions with rows in flight per warp.  Four take 64 registers, so 32 resident
// warps per multiprocessor in place of 48, and pay where few rows are copied (128 floats: 400,000 samples in four parts 124.5 -> 105 us,
// 1M in four 184 -> 176.5, 1M in 64 1,090 -> 1,020); two are better from where the rows fill more than two rounds of 32 warps
// (400,000 at once 66.6 -> 64.1, 1M 134.2 -> 129.7; in between, 240,000 at once 50.1 -> 50.5).
template <int C8, unsigned SHARERS, int UNR>
__global__ void __launch_bounds__(256)
lt_place_kernel(View v, HandleView h, uint64_t N, uint64_t cursor, uint64_t n, uint32_t q_first,
                uint32_t* __restrict__ out, const float* __restrict__ table, const float* slab,
                float* __restrict__ out_vals)
{
    grid_dependency_wait();
    const LtChunk c = lt_chunk(q_first + blockIdx.y, N, v.R, cursor, n);
    if (!c.active) return;
    const unsigned lane = threadIdx.x & 31;
    const uint4 pv = h.prev[c.q], wk = h.walk[c.q];
    const uint64_t oc = pv.x, ph = pv.y, pt = pv.z, end = oc + wk.x, tl = wk.y, cnt = wk.z;
    // the first warps take the words of the fresh entries that are walked, those after them the entries that earlier
    // calls postponed and this one emits (they come after the local ones)
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t w = warp / SHARERS;
    const unsigned share = (unsigned)(warp % SHARERS);
    const bool writes = share == 0;                                  // places are written down once
    const uint64_t words = wk.x ? ((end + 31) >> 5) - (oc >> 5) : 0;
    const uint64_t old = cnt < pt - ph ? cnt : pt - ph;
    uint32_t key = 0;
    bool emitted = false;
    uint32_t opos = 0;                                               // where the emitted key went
    if (w < words) {
        const uint64_t word = (oc >> 5) + w, i = word * 32 + lane;
        const bool walked = i >= oc && i < end;
        const uint32_t bits = h.flags[(c.b0 >> 5) + c.q + word];
        const uint64_t before = (uint64_t)h.prefix[(c.b0 >> 5) + c.q + word] + __popc(bits & ((1u << lane) - 1u));
        const bool loc = (bits >> lane) & 1u;
        if (walked) {
            key = h.keys[c.b0 + i];
            if (loc) {
                opos = (uint32_t)(c.out_base + before);
                if (writes) out[opos] = key;
                emitted = true;
            } else {
                // postponed: queued behind the non-local entries before it, emitted by this very call if the queue's
                // head gets that far, and moved to the worker.  (Locality was judged before any key moved: the bits
                // were all looked up by the kernel before this one.)
                const uint64_t at = pt + ((i - oc) - before);
                if (writes) h.post[c.b0 + at] = key;
                if (at >= ph && at < ph + cnt) {
                    opos = (uint32_t)(c.out_base + tl + (at - ph));
                    if (writes) out[opos] = key;
                    emitted = true;
                }
                if (writes) mark_localize(v, key, c.q);
            }
        }
    } else {
        const uint64_t j = (w - words) * 32 + lane;
        if ((w - words) * 32 >= old) return;
        if (j < old) {
            key = h.post[c.b0 + ph + j];
            opos = (uint32_t)(c.out_base + tl + j);
            if (writes) out[opos] = key;
            emitted = true;
        }
    }
    if (writes) count_sample(v, key, emitted);
    if (C8 > 0) {
        constexpr int RPI = C8 > 0 ? 32 / C8 : 1, ROWS = 32 / (int)SHARERS;      // rows per instruction; per warp
        static_assert(ROWS % (UNR * RPI) == 0, "whole turns");
        const unsigned sub = lane / (C8 > 0 ? C8 : 1), ch = lane % (C8 > 0 ? C8 : 1);
        const uint64_t L = (uint64_t)v.L4 * 4;
        const uint32_t src = emitted ? key : 0xFFFFFFFFu;
        uint32_t pend = 0xFFFFFFFFu;                                 // replica row of a replicated key
        if (emitted && key_is_hot(v, key)) pend = c.q * (uint32_t)v.Hcap + (uint32_t)__ldg(v.slot_of + key);
        for (int r1 = 0; r1 < ROWS; r1 += UNR * RPI) {
            const int r0 = (int)share * ROWS + r1;
            uint32_t so[UNR], po[UNR], oo[UNR];
            F8 a[UNR];
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                const int row = r0 + u * RPI + (int)sub;
                so[u] = __shfl_sync(0xFFFFFFFFu, src, row);
                po[u] = __shfl_sync(0xFFFFFFFFu, pend, row);
                oo[u] = __shfl_sync(0xFFFFFFFFu, opos, row);
            }
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                if (so[u] == 0xFFFFFFFFu) continue;
                const float* p = table + (uint64_t)so[u] * L + 8 * ch;
                a[u] = po[u] == 0xFFFFFFFFu ? ld8_stream(p) : ld8_cached(p);
                if (po[u] != 0xFFFFFFFFu) {
                    const F8 d = ld8_plain(slab + (uint64_t)po[u] * L + 8 * ch);
                    a[u].a = add4(a[u].a, d.a);
                    a[u].b = add4(a[u].b, d.b);
                }
            }
#pragma unroll
            for (int u = 0; u < UNR; ++u)
                if (so[u] != 0xFFFFFFFFu) st8_stream(out_vals + (uint64_t)oo[u] * L + 8 * ch, a[u]);
        }
    }
}

static nups_status pull_internal(nups_store* s, int id, uint64_t n, uint32_t* d_keys_out, float* d_vals_out,
                                 cudaStream_t st)
{
    Handle& h = s->handle[id];
    Dist& d = s->dist[h.dist];
    if (n > h.N - h.cursor) return NUPS_ESTATE;
    if (n == 0) return NUPS_OK;
    if (d.level == NUPS_LONGTERM) {
        nups_status rc = nups_new_epoch(s, st);
        if (rc != NUPS_OK) return rc;
    }
    View v = nups_view(s);
    HandleView hv = handle_view(h.buf, h.N, s->R, d.level);
    DrawParams p = draw_params(d);
    if (d.level == NUPS_LONGTERM) {
        // sub-handles overlapped by [cursor, cursor + n)
        uint32_t qf = 0, ql = 0;
        for (uint32_t q = 0; q < s->R; ++q) {
            uint64_t b0 = ((uint64_t)q * h.N) / s->R, b1 = ((uint64_t)(q + 1) * h.N) / s->R;
            if (b0 <= h.cursor && h.cursor < b1) qf = q;
            if (b0 <= h.cursor + n - 1 && h.cursor + n - 1 < b1) ql = q;
        }
        const uint64_t max_size = (h.N + s->R - 1) / s->R;
        // words of a sub-handle and of its postponed entries: together at most three more than the sub-handle's entries fill
        const dim3 by_word(grid_for(max_size / 32 + 4, 8), ql - qf + 1);
        // as many blocks as are resident at once: every block pays for a fence and a ticket
        const unsigned resident = (unsigned)s->sm_count * LT_BLOCKS / (ql - qf + 1);
        const unsigned walkers = grid_for(max_size / 32 + 2, LT_THREADS / 32, resident ? resident : 1);
        nups_launch_dependent(lt_walk_kernel, dim3(walkers, ql - qf + 1), LT_THREADS, 0, st, v, hv, h.N, h.cursor, n, qf);
        LAUNCH_CHECK(s);
        // the placement pass can copy the rows itself (one table of 64, 128 or 256 floats per row, 32-byte aligned output)
        const uint32_t c8 = s->L / 8;
        const bool fused = d_vals_out && s->vb == 4 && s->L % 8 == 0 && (c8 == 8 || c8 == 16 || c8 == 32) &&
                           ((uintptr_t)d_vals_out & 31) == 0 && (uint64_t)s->R * s->Hcap < 0xFFFFFFFFull;
        // warps per word: as many as are resident at once, 32 per multiprocessor
        unsigned sharers = 1;
        while (fused && sharers < 4 && (uint64_t)by_word.x * by_word.y * 8 * sharers * 2 <= (uint64_t)s->sm_count * 32) sharers *= 2;
        const dim3 shared_words(grid_for((max_size / 32 + 4) * sharers, 8), by_word.y);
        if (fused) nups_time_begin(s, st, NUPS_TIMED_SAMPLE_ROWS);
        const bool deep = n <= (uint64_t)s->sm_count * 32 * 64;         // rows in two rounds of resident warps, see lt_place_kernel
#define NUPS_PLACE(C8_, DEEP_)                                                                                            \
    nups_launch_dependent(sharers == 4 ? lt_place_kernel<C8_, 4, DEEP_> : sharers == 2 ? lt_place_kernel<C8_, 2, DEEP_>   \
                          : deep ? lt_place_kernel<C8_, 1, DEEP_> : lt_place_kernel<C8_, 1, 2>, shared_words, 256, 0, st, v, hv, h.N, \
                          h.cursor, n, qf, d_keys_out, s->val, s->dval, d_vals_out)
        if (fused && c8 == 8) NUPS_PLACE(8, 2);
        else if (fused && c8 == 16) NUPS_PLACE(16, 4);
        else if (fused) NUPS_PLACE(32, 4);
#undef NUPS_PLACE
        else nups_launch_dependent(lt_place_kernel<0, 1, 1>, by_word, 256, 0, st, v, hv, h.N, h.cursor, n, qf, d_keys_out, nullptr, nullptr, nullptr);
        if (fused) nups_time_end(s, st);
        LAUNCH_CHECK(s);
        if (fused) {
            h.cursor += n;
            if (h.cursor == h.N) h.used = 0;
            return NUPS_OK;
        }
    } else if (d_vals_out && d.level != NUPS_NONCONFORM && !s->cfg.count_accesses) {
        // keys fixed at PrepareSample and nothing to count: the row gather reads them from the handle and hands them out
        // on its way, which saves a launch
        h.cursor += n;
        if (h.cursor == h.N) h.used = 0;
        return nups_gather_internal(s, hv.keys + (h.cursor - n), n, d_vals_out, nullptr, 1, h.cursor - n, h.N, 0, st, d_keys_out);
    } else {
        nups_launch_dependent(emit_kernel, grid_for(n, 256), 256, 0, st, v, p, hv, h.N, h.cursor, n, d.level == NUPS_NONCONFORM, d_keys_out);
        LAUNCH_CHECK(s);
    }
    if (d_vals_out) {
        nups_status rc = nups_gather_internal(s, d_keys_out, n, d_vals_out, nullptr, 1, h.cursor, h.N, 0, st, nullptr);
        if (rc != NUPS_OK) return rc;
    }
    h.cursor += n;
    if (h.cursor == h.N) h.used = 0;       // released; the buffer stays for the next handle
    return NUPS_OK;
}

extern "C" nups_status nups_pull_sample(nups_store* s, nups_handle handle, uint64_t n, uint32_t* d_keys_out,
                                        void* d_vals_out, void* stream)
{
    if (!s || handle < 0 || handle >= NUPS_MAX_HANDLES || !s->handle[handle].used) return NUPS_EINVAL;
    if (n && !d_keys_out) return NUPS_EINVAL;
    return pull_internal(s, (int)handle, n, d_keys_out, (float*)d_vals_out, (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------------------------
// PrepareSample + one full PullSample (keys only) in a single launch, for the workload steps: the
// same keys as the handle path gives, written straight to `out`.  Stream offsets are read from one
// half of the distribution's offset array and the advanced offsets written to the other half.
// ---------------------------------------------------------------------------------------------
// blockIdx.y (iid) / blockIdx.z (reuse) = batch: `batches` handles of N samples each are drawn back to back,
// exactly as that many separate calls would draw them; batch b goes to out + b * N.
__global__ void draw_direct_iid_kernel(View v, DrawParams p, const unsigned long long* __restrict__ off_cur,
                                       unsigned long long* __restrict__ off_next, uint64_t N, uint32_t batches,
                                       int local_only, int localize, uint32_t* __restrict__ out)
{
    grid_dependency_wait();
    const uint64_t o = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t bt = blockIdx.y;
    const bool in = o < N;
    uint32_t k = 0, q = 0;
    out += (uint64_t)bt * N;
    if (in) {
        q = chunk_of_pos(o, N, v.R);
        const unsigned long long size = chunk_begin(q + 1, N, v.R) - chunk_begin(q, N, v.R);
        k = draw_iid(p, q, off_cur[q] + (unsigned long long)bt * size + (o - chunk_begin(q, N, v.R)));
    }
    if (local_only) k = first_local_warp(v, p, q, k, in);
    const bool repeats = localize && __popc(__match_any_sync(0xFFFFFFFFu, in ? k : 0xFFFFFFFFu - (threadIdx.x & 31))) > 1;
    if (in) {
        out[o] = k;
        if (localize) mark_localize_rare(v, k, q, repeats);
    }
    count_sample(v, k, in);
    if (blockIdx.x == 0 && blockIdx.y == 0)
        for (uint32_t w = threadIdx.x; w < v.R; w += blockDim.x)
            off_next[w] = off_cur[w] + (unsigned long long)batches * (chunk_begin(w + 1, N, v.R) - chunk_begin(w, N, v.R));
}

__global__ void draw_direct_reuse_kernel(View v, DrawParams p, const unsigned long long* __restrict__ off_cur,
                                         unsigned long long* __restrict__ off_next, uint64_t N, uint32_t batches,
                                         int localize, uint32_t* __restrict__ out, uint32_t T)
{
    grid_dependency_wait();
    const uint32_t q = blockIdx.y, R = v.R;
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0)
        for (uint32_t w = threadIdx.x; w < R; w += blockDim.x)
            off_next[w] = off_cur[w] + (unsigned long long)batches * (chunk_begin(w + 1, N, R) - chunk_begin(w, N, R));
    const unsigned long long b0 = chunk_begin(q, N, R), size = chunk_begin(q + 1, N, R) - b0;
    if (size == 0) return;
    out += (uint64_t)blockIdx.z * N;
    const unsigned long long s0 = off_cur[q] + (unsigned long long)blockIdx.z * size;
    reuse_pool_visit(p, q, s0, s0 + size, T, [&](bool in, uint32_t k, unsigned long long rel, bool mark) {
        if (in) {
            out[b0 + rel] = k;
            if (localize && mark) mark_localize(v, k, q);
        }
        count_sample(v, k, in);
    }, [&](uint32_t k) { if (localize) mark_localize(v, k, q); });
}

// Sample-ahead for the workload steps.  The sample streams are a pure function of (seed, worker,
// position), so the negatives of the next NUPS_SAMPLE_AHEAD steps can be drawn in one launch and
// handed out one batch per step.  If anything else touches the distribution before they are used up
// (PrepareSample, a step with another size), the stream offsets are rewound by what was not handed out,
// so every sample sequence is the same as without sample-ahead.  Only used where drawing early has no
// other effect: fast mode, no access counting, no ownership tracking.
__global__ void rewind_kernel(unsigned long long* off, uint64_t N, uint32_t R, uint32_t batches)
{
    const uint32_t q = threadIdx.x;
    if (q < R) off[q] -= (unsigned long long)batches * (chunk_begin(q + 1, N, R) - chunk_begin(q, N, R));
}

nups_status nups_sample_ahead_rewind(nups_store* s, cudaStream_t st)
{
    if (s->ahead_dist < 0) return NUPS_OK;
    const uint32_t left = s->ahead_total - s->ahead_next;
    if (left) {
        Dist& d = s->dist[s->ahead_dist];
        rewind_kernel<<<1, 256, 0, st>>>(d.off + (size_t)d.cur * s->R, s->ahead_N, s->R, left);
        LAUNCH_CHECK(s);
    }
    s->ahead_dist = -1;
    return NUPS_OK;
}

// negatives of a workload step: one handle of N samples, pulled at once into library memory
nups_status nups_draw_negatives(nups_store* s, int32_t dist, uint64_t N, cudaStream_t st)
{
    s->last_negs_n = 0;
    if (N == 0) return NUPS_OK;
    if (dist < 0 || dist >= NUPS_MAX_DISTS || !s->dist[dist].used || N >= (1ull << 32)) return NUPS_EINVAL;
    // a batch drawn ahead for exactly this request?
    if (s->ahead_dist == dist && s->ahead_N == N && s->ahead_next < s->ahead_total) {
        s->last_negs = s->negs_buf + (uint64_t)s->ahead_next * N;
        s->last_negs_n = N;
        s->ahead_next++;
        return NUPS_OK;
    }
    nups_status rc = nups_sample_ahead_rewind(s, st);
    if (rc != NUPS_OK) return rc;
    Dist& d = s->dist[dist];
    const bool plain = d.level == NUPS_CONFORM || d.level == NUPS_BOUNDED;
    const uint32_t batches = (plain && !s->cfg.deterministic && !s->cfg.count_accesses && !s->own &&
                              N * NUPS_SAMPLE_AHEAD < (1ull << 28)) ? NUPS_SAMPLE_AHEAD : 1;
    if (N * batches > s->negs_cap) {
        uint64_t want = N * batches + N / 4;
        if (s->dev_cap && (want * 4 > s->dev_cap || s->dev_bytes - s->negs_cap * 4 > s->dev_cap - want * 4)) return NUPS_ENOMEM;
        nups_dev_free(s, s->negs_buf, s->negs_cap * 4);
        s->negs_buf = nullptr; s->negs_cap = 0;
        rc = nups_dev_alloc(s, (void**)&s->negs_buf, want * 4);
        if (rc != NUPS_OK) return rc;
        s->negs_cap = want;
    }
    s->last_negs = s->negs_buf;
    if (d.level == NUPS_LONGTERM) {
        // postponing needs the handle's walk state: PrepareSample, then one full PullSample
        int id = -1;
        rc = prepare_internal(s, dist, N, &id, st);
        if (rc != NUPS_OK) return rc;
        rc = pull_internal(s, id, N, s->last_negs, nullptr, st);
        if (rc != NUPS_OK) return rc;
        s->last_negs_n = N;
        return NUPS_OK;
    }
    const int localize = s->own && d.level != NUPS_NONCONFORM;
    if (localize) {
        rc = nups_new_epoch(s, st);
        if (rc != NUPS_OK) return rc;
    }
    View v = nups_view(s);
    DrawParams p = draw_params(d);
    const unsigned long long* off_cur = d.off + (size_t)d.cur * s->R;
    unsigned long long* off_next = d.off + (size_t)(d.cur ^ 1) * s->R;
    if (d.level == NUPS_BOUNDED) {
        const ReuseShape sh = reuse_shape(d.U, d.G);
        nups_launch_dependent(draw_direct_reuse_kernel, dim3(reuse_pools((N + s->R - 1) / s->R, d.U, d.G), s->R, batches),
                              REUSE_THREADS, sh.smem, st, v, p, off_cur, off_next, N, batches, localize, s->negs_buf, sh.T);
    } else {
        nups_launch_dependent(draw_direct_iid_kernel, dim3(grid_for(N, 256), batches), 256, 0, st, v, p, off_cur, off_next, N, batches,
                                                                              d.level == NUPS_NONCONFORM, localize,
                                                                              s->negs_buf);
    }
    LAUNCH_CHECK(s);
    d.cur ^= 1;
    s->last_negs_n = N;
    if (batches > 1) {
        s->ahead_dist = dist; s->ahead_N = N; s->ahead_total = batches; s->ahead_next = 1;
    }
    return NUPS_OK;
}

extern "C" nups_status nups_last_negatives(nups_store* s, const uint32_t** h_d_keys_out, uint64_t* h_n_out)
{
    if (!s || !h_d_keys_out || !h_n_out) return NUPS_EINVAL;
    *h_d_keys_out = s->last_negs;
    *h_n_out = s->last_negs_n;
    return NUPS_OK;
}

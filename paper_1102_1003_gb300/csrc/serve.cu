// Serving: a device-resident pool of sets answering intersection-size and
// conjunctive queries (Sec. I: a conjunctive query is a set intersection),
// with a continuous-batching request loop.
//
// Pool storage.  Every set keeps its sorted tidlist.  Sets for which the 8-bit
// BatMap is compact (|S| >= r_0 / c, Sec. III-A: compression pays only when
// the set is dense enough) also get a BatMap, built by the same GPU build as
// pair mining.  A query |S_a1 cap ... cap S_ak| enumerates the smallest set
// and counts the elements present in every other set (the k-way counting idea
// of Sec. V): membership in a BatMap is two byte probes -- x is stored in two
// of the three tables, so tables 1 and 2 always hold at least one copy -- plus
// a binary search of the set's failed insertions; a set without a BatMap is
// searched in two levels: a sampled index of every IDX_STRIDE-th tid of each
// set (1/64 of the tidlists, small enough that its upper levels stay in L2)
// narrows the search to one block of IDX_STRIDE tids (256 contiguous bytes).
// Where the other set is not much larger than the smallest one, its tids between
// a task's first and last element are read once instead, whichever form it has.
//
// Work is cut into tasks of up to 512 elements of the smallest set; one warp
// runs a task.
#include <algorithm>
#include <chrono>
#include <memory>
#include <cstring>
#include <thread>

#include "common.cuh"
#include "perm.cuh"
#include "scan.cuh"

namespace bm {

void build_set(batmap_set *S, const uint64_t *d_offsets, const uint32_t *d_tids, const uint32_t *d_perm);

constexpr uint32_t TASK_ELEMS = 512;
constexpr uint32_t MAX_K = 8;
constexpr uint32_t IDX_STRIDE = 64;  // tids per block of the sampled index

struct QueryDesc {
    uint32_t k;
    uint32_t ids[MAX_K];  // smallest set first
};
struct ProbeTask {
    uint32_t q;      // query index within the batch
    uint32_t begin;  // element range of the smallest set
    uint32_t end;
};

struct PoolView {
    const uint64_t *off;      // [n+1] CSR of all sets
    const uint32_t *tids;
    PermView perm;            // pi_0 .. pi_2 (the caller's table or computed)
    const int32_t *bm_index;  // [n] index among BatMap-backed sets or -1
    const uint64_t *bm_base;  // [nb] byte offset of the BatMap
    const uint32_t *bm_rlog;  // [nb] log2 r
    const uint64_t *f_off;    // [nb+1] failed insertions per BatMap-backed set
    const uint32_t *f_tid;
    const uint8_t *bm;        // BatMap bytes
    uint32_t m, shift;
    const uint64_t *idx_off;  // [n+1] sampled index: ceil(|S_c| / IDX_STRIDE) entries per set
    const uint32_t *idx;      // entry j of set c = tid IDX_STRIDE * j of set c
};

// ---- one task: the elements of a range of the smallest set that all others hold ----
// A warp keeps the task's elements in shared memory and one bit per element in
// registers: bit j of a lane's word is element 32 j + lane.
//
// Against one more set, whose tids between the task's first and last element
// ("window") are found by two 32-way searches of the sampled index:
// stream: the window goes through shared memory once, PART tids at a time with the
//   next on their way; the elements up to a chunk's last tid are searched in it,
//   four of a lane at once.  Where the window has up to STREAM tids per element.
// search: each element by itself, four of a lane at once: a sample of the window's
//   index entries in shared memory, then at most the block of IDX_STRIDE tids.
// bytes: sets with a BatMap, two byte probes and the failed insertions.
// Bound: instruction issue (56% of it at 24% occupancy) and the latency of a task's
// first reads.  4096 queries over 4000 sets of 10..10^6 tids (51 M elements, 0.6 GB of
// windows), a call: 1200 us with one element at a time, its 20 dependent reads 32
// times in a row; 610 us; 540 us with shorter tasks in smaller blocks (here).  STREAM 4,
// 8, 16, 32, 64: 803, 691, 629, 610, 620 us.  The lists of 256: 874 -> 245 us, as the
// write pass probed again and the binding called twice.
constexpr uint32_t PROBE_WARPS = 2, WIN = 512, PART = 512;
constexpr uint32_t STREAM = 32;

struct ProbeShared {
    uint32_t x[TASK_ELEMS + 4];  // from a 16-byte boundary of the set on
    union {
        uint32_t chunk[2][PART];  // stream
        uint32_t win[WIN];         // search
    };
};

// 16-byte asynchronous copies of p's `quads` quads by a warp, one group.
__device__ __forceinline__ void copy_quads(uint32_t *to, const uint32_t *from, uint32_t quads, uint32_t lane) {
    for (uint32_t q = lane; q < quads; q += 32)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to + 4 * q)),
                     "l"(from + 4 * q)
                     : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void copies_wait() {  // all but the last N groups are there
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
    __syncwarp();
}

// Numbers of entries <= v0 and <= v1 of the ascending a[0..n), by a warp.
__device__ __forceinline__ void count_le(const uint32_t *__restrict__ a, uint32_t n, uint32_t v0, uint32_t v1,
                                         uint32_t lane, uint32_t &c0, uint32_t &c1) {
    uint32_t lo[2] = {0, 0}, hi[2] = {n, n};
    const uint32_t v[2] = {v0, v1};
    while (hi[0] - lo[0] || hi[1] - lo[1]) {
        uint32_t x[2], at[2];
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const uint32_t span = hi[q] - lo[q];
            at[q] = span > 32 ? (uint32_t)((uint64_t)span * (lane + 1) / 33) : lane;  // ascending, < span (or no lane)
            x[q] = at[q] < span ? __ldg(&a[lo[q] + at[q]]) : 0xffffffffu;
        }
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const uint32_t span = hi[q] - lo[q];
            const uint32_t c = __popc(__ballot_sync(0xffffffffu, at[q] < span && x[q] <= v[q]));
            const uint32_t below = __shfl_sync(0xffffffffu, at[q], c ? c - 1 : 0);
            const uint32_t above = __shfl_sync(0xffffffffu, at[q], c < 32 ? c : 31);
            if (!span) continue;
            if (c < 32 && above < span) hi[q] = lo[q] + above;
            if (c) lo[q] += below + 1;
        }
    }
    c0 = lo[0];
    c1 = lo[1];
}

// x: the task's n elements, of which [from, to) of the tids may hold some.
__device__ __forceinline__ uint32_t stream_members(const PoolView &P, ProbeShared &S, const uint32_t *x, uint32_t n,
                                                   uint32_t alive, uint64_t from, uint64_t to, uint32_t lane) {
    const uint32_t rows = (n + 31) / 32, top = x[n - 1];
    uint32_t kept = 0, row = 0, skip = (uint32_t)(from & 3);
    int32_t past = -1;  // (tids are below 2^30) the last tid of the chunk before
    // chunks lie on 16-byte boundaries (the tids have room up to a multiple of 4)
    const uint32_t *p = P.tids + (from - skip);
    uint64_t left = to - (from - skip);
    auto quads = [](uint64_t tids) { return (uint32_t)(min(tids, (uint64_t)PART) + 3) / 4; };
    copy_quads(S.chunk[0], p, quads(left), lane);
    for (uint32_t c = 0; left; c ^= 1) {
        const uint32_t len = (uint32_t)min(left, (uint64_t)PART);
        left -= len;
        p += PART;
        copy_quads(S.chunk[c ^ 1], p, left ? quads(left) : 0, lane);
        copies_wait<1>();
        const uint32_t *s = S.chunk[c] + skip, count = len - skip, last = s[count - 1];
        skip = 0;
        const uint32_t upto = __popc(__ballot_sync(0xffffffffu, lane < rows && x[min(32 * lane, n - 1)] <= last));
        const uint32_t p2 = 1u << (31 - __clz(count));
        for (uint32_t j = row; j < upto; j += 4) {
            uint32_t v[4], at[4], want = 0;
#pragma unroll
            for (int u = 0; u < 4; u++) {
                v[u] = x[min(32 * (j + u) + lane, n - 1)];
                at[u] = 0;
                if (j + u < upto && v[u] <= last && (int32_t)v[u] > past) want |= 1u << u;
            }
            want &= alive >> j;  // (no bits from n on)
            if (!__any_sync(0xffffffffu, want)) continue;
            for (uint32_t step = p2; step; step >>= 1)
#pragma unroll
                for (int u = 0; u < 4; u++)
                    if (at[u] + step < count && s[at[u] + step] <= v[u]) at[u] += step;
#pragma unroll
            for (int u = 0; u < 4; u++)
                if ((want >> u & 1u) && s[at[u]] == v[u]) kept |= 1u << (j + u);
        }
        __syncwarp();
        if (last >= top) break;
        past = (int32_t)last;
        row = upto ? upto - 1 : 0;
    }
    copies_wait<0>();
    return kept;
}

// from, win: the index entries that elements may follow (entry from - 1, if any, is <= all).
__device__ __forceinline__ uint32_t search_members(const PoolView &P, ProbeShared &S, const uint32_t *xs, uint32_t alive, uint32_t c,
                                                   uint32_t from, uint32_t win, uint32_t lane) {
    const uint64_t b = P.off[c];
    const uint32_t size = (uint32_t)(P.off[c + 1] - b);  // <= 2^30
    const uint32_t *idx = P.idx + P.idx_off[c] + from, *tids = P.tids + b;
    const uint32_t every = win > WIN ? (win + WIN - 1) / WIN : 1, ns = win / every;  // samples, <= WIN
    for (uint32_t i = lane; i < ns; i += 32) S.win[i] = __ldg(&idx[(i + 1) * every - 1]);
    __syncwarp();
    const uint32_t s2 = ns ? 1u << (31 - __clz(ns)) : 0, e2 = every > 1 ? 1u << (31 - __clz(every - 1)) : 0;
    uint32_t kept = 0;
    for (uint32_t left = alive; __any_sync(0xffffffffu, left != 0);) {
        uint32_t bit[4], x[4], lo[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            bit[u] = left & (0u - left);
            left &= left - 1;
            x[u] = bit[u] ? xs[32 * (__ffs(bit[u]) - 1) + lane] : 0;
            lo[u] = 0;
        }
        for (uint32_t step = s2; step; step >>= 1)  // samples <= x
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (lo[u] + step <= ns && S.win[lo[u] + step - 1] <= x[u]) lo[u] += step;
#pragma unroll
        for (int u = 0; u < 4; u++) lo[u] *= every;
        uint32_t end[4];
#pragma unroll
        for (int u = 0; u < 4; u++) end[u] = min(win, lo[u] + every - 1);
        for (uint32_t step = e2; step; step >>= 1)  // entries of the window <= x
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (bit[u] && lo[u] + step <= end[u] && __ldg(&idx[lo[u] + step - 1]) <= x[u]) lo[u] += step;
        uint32_t at[4], top[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {  // the block of tids whose first is the last entry <= x
            const uint32_t e = from + lo[u];
            if (!e) bit[u] = 0;  // below the set's first tid
            at[u] = e ? IDX_STRIDE * (e - 1) : 0;
            top[u] = min(size, at[u] + IDX_STRIDE);
        }
#pragma unroll
        for (uint32_t step = IDX_STRIDE / 2; step; step >>= 1)
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (bit[u] && at[u] + step < top[u] && __ldg(&tids[at[u] + step]) <= x[u]) at[u] += step;
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (bit[u] && __ldg(&tids[at[u]]) == x[u]) kept |= bit[u];
    }
    __syncwarp();
    return kept;
}

__device__ __forceinline__ bool bsearch_u32(const uint32_t *a, uint64_t lo, uint64_t hi, uint32_t x) {
    while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        const uint32_t v = a[mid];
        if (v == x) return true;
        if (v < x) lo = mid + 1; else hi = mid;
    }
    return false;
}

__device__ __forceinline__ uint32_t byte_members(const PoolView &P, const uint32_t *xs, uint32_t alive, uint32_t b,
                                                 uint32_t lane) {
    const uint8_t *bm = P.bm + P.bm_base[b];
    const uint32_t r = 1u << P.bm_rlog[b];
    const uint64_t f0 = P.f_off[b], f1 = P.f_off[b + 1];
    uint32_t kept = 0;
    for (uint32_t left = alive; left;) {
        uint32_t bit[4], x[4], want[4][2], got[4][2];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            bit[u] = left & (0u - left);
            left &= left - 1;
            x[u] = bit[u] ? xs[32 * (__ffs(bit[u]) - 1) + lane] : 0;
#pragma unroll
            for (uint32_t t = 0; t < 2; t++) {
                const uint32_t pi = P.perm(t, x[u]);
                want[u][t] = (pi >> P.shift) + 1u;
                got[u][t] = bit[u] ? __ldg(&bm[slot_of(t, pi, r, P.shift)]) & 0x7Fu : 0;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (bit[u] && (got[u][0] == want[u][0] || got[u][1] == want[u][1] || bsearch_u32(P.f_tid, f0, f1, x[u]))) kept |= bit[u];
    }
    __syncwarp();
    return kept;
}

__device__ __forceinline__ uint32_t probe_task(const PoolView &P, const QueryDesc &Q, const ProbeTask &tk, ProbeShared &S,
                                               uint32_t lane) {
    const uint32_t n = tk.end - tk.begin, mine = n > lane ? (n - lane + 31) / 32 : 0;
    uint32_t alive = mine == 32 ? 0xffffffffu : (1u << mine) - 1;
    if (Q.k == 1) return alive;
    const uint64_t a0 = P.off[Q.ids[0]] + tk.begin;
    const uint32_t skip = (uint32_t)(a0 & 3), *x = S.x + skip;
    copy_quads(S.x, P.tids + (a0 - skip), (n + skip + 3) / 4, lane);
    const uint32_t first = __ldg(&P.tids[a0]), last = __ldg(&P.tids[a0 + n - 1]);
    bool there = false;
    for (uint32_t t = 1; t < Q.k; t++) {
        const uint32_t todo = __reduce_add_sync(0xffffffffu, __popc(alive));
        if (!todo) break;
        const uint32_t c = Q.ids[t];
        const uint64_t b = P.off[c], e = P.off[c + 1];
        uint32_t c0 = 0, c1 = 0;
        uint64_t from = b, to = e;
        // (a set of one chunk is read whole: the search for the window would take longer, 54.2 -> 53.2 ms
        // one by one in the pool above HOST_TASKS)
        if (e - b > PART || e - b > (uint64_t)STREAM * todo) {
            const uint64_t i0 = P.idx_off[c];
            count_le(P.idx + i0, (uint32_t)(P.idx_off[c + 1] - i0), first, last, lane, c0, c1);
            from = b + (uint64_t)IDX_STRIDE * (c0 ? c0 - 1 : 0);
            to = min(e, b + (uint64_t)IDX_STRIDE * c1);
        }
        const int32_t bm = P.bm_index[c];
        if (!there) copies_wait<0>();
        there = true;
        if (to <= from) return 0;  // all are below its first tid, or there is none
        if (to - from <= (uint64_t)STREAM * todo) alive = stream_members(P, S, x, n, alive, from, to, lane);
        else if (bm >= 0) alive = byte_members(P, x, alive, (uint32_t)bm, lane);
        else alive = search_members(P, S, x, alive, c, c0, c1 - c0, lane);
    }
    return alive;
}

// The tasks of each query, a block each.
__global__ void k_query_tasks(const uint64_t *__restrict__ off, const QueryDesc *__restrict__ qs,
                              const uint32_t *__restrict__ first, uint32_t elems, ProbeTask *__restrict__ tasks) {
    const uint32_t q = blockIdx.x, t0 = first[q], n = first[q + 1] - t0, a = qs[q].ids[0];
    const uint32_t size = (uint32_t)(off[a + 1] - off[a]);
    for (uint32_t k = threadIdx.x; k < n; k += blockDim.x) tasks[t0 + k] = {q, k * elems, min(size, (k + 1) * elems)};
}

// One warp a task.  Counts: added to the query's.  Lists (masks not NULL): the
// task's count and its words, which the write pass after an exclusive scan over
// tasks ranks in element order, so every answer is ascending.
__global__ void __launch_bounds__(32 * PROBE_WARPS)
k_probe(PoolView P, const QueryDesc *__restrict__ qs, const ProbeTask *__restrict__ tasks, uint32_t ntasks,
        unsigned long long *__restrict__ counts, uint64_t *__restrict__ task_counts, uint32_t *__restrict__ masks) {
    __shared__ __align__(16) ProbeShared shared[PROBE_WARPS];
    const uint32_t lane = threadIdx.x & 31, w = blockIdx.x * PROBE_WARPS + (threadIdx.x >> 5);
    if (w >= ntasks) return;
    const ProbeTask tk = tasks[w];
    const uint32_t alive = probe_task(P, qs[tk.q], tk, shared[threadIdx.x >> 5], lane);
    const uint32_t cnt = __reduce_add_sync(0xffffffffu, __popc(alive));
    if (masks) masks[32ull * w + lane] = alive;
    if (lane) return;
    if (task_counts) task_counts[w] = cnt;
    else if (cnt) atomicAdd(&counts[tk.q], (unsigned long long)cnt);
}

__global__ void k_probe_write(PoolView P, const QueryDesc *__restrict__ qs, const ProbeTask *__restrict__ tasks,
                              uint32_t ntasks, const uint64_t *__restrict__ task_off, const uint32_t *__restrict__ masks,
                              uint32_t *__restrict__ out, uint64_t cap) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= ntasks) return;
    const uint32_t mine = masks[32ull * w + lane];
    if (!__any_sync(0xffffffffu, mine != 0)) return;
    const ProbeTask tk = tasks[w];
    const uint32_t *a = P.tids + P.off[qs[tk.q].ids[0]] + tk.begin;
    uint64_t running = task_off[w];
    for (uint32_t j = 0; j < 32; j++) {
        const uint32_t mask = __ballot_sync(0xffffffffu, mine >> j & 1u);
        const uint64_t pos = running + __popc(mask & ((1u << lane) - 1u));
        if ((mine >> j & 1u) && pos < cap) out[pos] = a[32 * j + lane];
        running += __popc(mask);
    }
}

__global__ void k_query_offsets(const uint64_t *__restrict__ task_off, const uint32_t *__restrict__ first_task,
                                uint32_t nq, uint64_t *__restrict__ out_off) {
    const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q <= nq) out_off[q] = task_off[first_task[q]];
}

// The sampled index: entry j of set c is tid IDX_STRIDE * j of set c.
__global__ void k_sample_index(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tids, uint32_t n,
                               const uint64_t *__restrict__ idx_off, uint32_t *__restrict__ idx) {
    for (uint32_t c = blockIdx.x; c < n; c += gridDim.x) {
        const uint64_t b = off[c], k0 = idx_off[c], nk = idx_off[c + 1] - k0;
        for (uint64_t j = threadIdx.x; j < nk; j += blockDim.x) idx[k0 + j] = tids[b + (uint64_t)IDX_STRIDE * j];
    }
}

// One warp per set: every tid < m and strictly increasing within its set.
__global__ void k_validate_sets(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tids, uint32_t n,
                                uint32_t m, int *err) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < n; c += warps) {
        const uint64_t b = off[c], e = off[c + 1];
        bool bad = e < b;
        for (uint64_t i = b + lane; i < e && !bad; i += 32) {
            const uint32_t x = tids[i];
            bad = x >= m || (i + 1 < e && !(x < tids[i + 1]));
        }
        if (bad) atomicExch(err, 1);
    }
}

}  // namespace bm

using namespace bm;

struct batmap_pool {
    uint32_t m = 0, n = 0;
    std::vector<uint64_t> h_off;
    DevBuf<uint64_t> d_off;
    DevBuf<uint32_t> d_tids, d_perm;
    DevBuf<int32_t> d_bm_index;
    DevBuf<uint64_t> d_bm_base, d_fail_off;
    DevBuf<uint32_t> d_bm_rlog, d_fail_tid;
    DevBuf<uint8_t> d_bm;
    DevBuf<uint64_t> d_idx_off;  // sampled index of the tidlists
    DevBuf<uint32_t> d_idx;
    uint32_t n_big = 0, shift = 0;
    uint64_t bm_bytes = 0, n_failed = 0;
    PoolView view{};
};

namespace bm {

static void pool_create(const batmap_params *p, uint32_t m, uint32_t n, const uint64_t *d_offsets,
                        const uint32_t *d_tids, const uint32_t *d_perm, cudaStream_t st, batmap_pool **out) {
    BM_REQUIRE(out, BATMAP_ERR_ARG, "out is NULL");
    BM_REQUIRE(m >= 1 && m <= (1u << 30), BATMAP_ERR_ARG, "m must be in [1, 2^30]");
    batmap_params P;
    batmap_default_params(&P);
    if (p) P = *p;
    auto pool = std::make_unique<batmap_pool>();
    pool->m = m;
    pool->n = n;
    pool->h_off.assign(n + 1, 0);
    if (n) {
        BM_REQUIRE(d_offsets, BATMAP_ERR_ARG, "d_offsets is NULL");
        BM_CUDA(cudaMemcpyAsync(pool->h_off.data(), d_offsets, (n + 1) * 8ull, cudaMemcpyDeviceToHost, st));
        BM_CUDA(cudaStreamSynchronize(st));
    }
    const uint64_t T = pool->h_off[n];
    pool->d_off.alloc(n + 1);
    pool->d_tids.alloc((T + 3) / 4 * 4);  // read 16 bytes at a time
    if (d_perm) pool->d_perm.alloc(3ull * m);  // computed permutations need no table
    if (n) BM_CUDA(cudaMemcpyAsync(pool->d_off.p, d_offsets, (n + 1) * 8ull, cudaMemcpyDeviceToDevice, st));
    if (T) BM_CUDA(cudaMemcpyAsync(pool->d_tids.p, d_tids, T * 4ull, cudaMemcpyDeviceToDevice, st));
    if (d_perm) BM_CUDA(cudaMemcpyAsync(pool->d_perm.p, d_perm, 3ull * m * 4, cudaMemcpyDeviceToDevice, st));
    if (n) {
        DevBuf<int> err(1);
        BM_CUDA(cudaMemsetAsync(err.p, 0, sizeof(int), st));
        k_validate_sets<<<(unsigned)std::min<uint64_t>((n + 7) / 8, 65535), 256, 0, st>>>(pool->d_off.p,
                                                                                          pool->d_tids.p, n, m, err.p);
        BM_CHECK_LAUNCH();
        int h = 0;
        BM_CUDA(cudaMemcpyAsync(&h, err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
        BM_CUDA(cudaStreamSynchronize(st));
        BM_REQUIRE(h == 0, BATMAP_ERR_ARG, "tids must be strictly increasing per set and < m");
    }

    // the sampled index of every tidlist (all sets: BatMap-backed ones keep it too)
    {
        std::vector<uint64_t> ioff(n + 1, 0);
        for (uint32_t i = 0; i < n; i++)
            ioff[i + 1] = ioff[i] + (pool->h_off[i + 1] - pool->h_off[i] + IDX_STRIDE - 1) / IDX_STRIDE;
        pool->d_idx_off.alloc(n + 1);
        pool->d_idx.alloc(std::max<uint64_t>(ioff[n], 1));
        BM_CUDA(cudaMemcpyAsync(pool->d_idx_off.p, ioff.data(), (n + 1) * 8ull, cudaMemcpyHostToDevice, st));
        if (ioff[n]) {
            k_sample_index<<<(unsigned)std::min<uint32_t>(std::max<uint32_t>(n, 1), 65535), 256, 0, st>>>(
                pool->d_off.p, pool->d_tids.p, n, pool->d_idx_off.p, pool->d_idx.p);
            BM_CHECK_LAUNCH();
        }
    }

    // sets whose 8-bit BatMap is compact: c |S| >= r_0
    uint32_t shift = P.min_shift;
    while ((uint64_t)m > 127ull << shift) shift++;
    const uint64_t r0 = 1ull << shift;
    std::vector<int32_t> bm_index(n, -1);
    std::vector<uint32_t> big_ids;
    std::vector<uint64_t> sub_off(1, 0);
    for (uint32_t i = 0; i < n; i++) {
        const uint64_t sz = pool->h_off[i + 1] - pool->h_off[i];
        if (sz && (uint64_t)P.load_num * sz >= r0 * P.load_den) {
            bm_index[i] = (int32_t)big_ids.size();
            big_ids.push_back(i);
            sub_off.push_back(sub_off.back() + sz);
        }
    }
    const uint32_t nb = (uint32_t)big_ids.size();
    pool->n_big = nb;
    pool->d_bm_index.alloc(std::max<uint32_t>(n, 1));
    if (n) BM_CUDA(cudaMemcpyAsync(pool->d_bm_index.p, bm_index.data(), n * 4ull, cudaMemcpyHostToDevice, st));
    std::vector<uint64_t> base(nb);
    std::vector<uint32_t> rlog(nb);
    std::vector<uint64_t> f_off(nb + 1, 0);
    if (nb) {
        // BatMap bytes of every big set (same sizing rule as the build)
        uint64_t total_bytes = 0;
        std::vector<uint64_t> bytes_of(nb);
        for (uint32_t b = 0; b < nb; b++) {
            const uint64_t sz = sub_off[b + 1] - sub_off[b];
            const uint64_t need = (P.load_num * sz + P.load_den - 1) / P.load_den;
            uint64_t r = 1;
            while (r < need) r <<= 1;
            bytes_of[b] = 3 * std::max<uint64_t>(r, r0);
            total_bytes += bytes_of[b];
        }
        pool->d_bm.alloc(total_bytes);
        std::vector<uint32_t> f_chunks_tid;
        uint64_t bm_pos = 0, f_pos = 0;
        // build in chunks of at most ~4 GB of BatMaps, as each is built beside its copy in the pool
        for (uint32_t c0 = 0; c0 < nb;) {
            uint32_t c1 = c0;
            uint64_t cb = 0;
            while (c1 < nb && (c1 == c0 || cb + bytes_of[c1] <= (4ull << 30))) cb += bytes_of[c1++];
            const uint32_t cn = c1 - c0;
            std::vector<uint64_t> coff(cn + 1, 0);
            for (uint32_t j = 0; j < cn; j++) coff[j + 1] = coff[j] + (sub_off[c0 + j + 1] - sub_off[c0 + j]);
            DevBuf<uint64_t> s_off(cn + 1);
            DevBuf<uint32_t> s_tids(coff[cn]);
            BM_CUDA(cudaMemcpyAsync(s_off.p, coff.data(), (cn + 1) * 8ull, cudaMemcpyHostToDevice, st));
            for (uint32_t j = 0; j < cn; j++) {
                const uint32_t i = big_ids[c0 + j];
                BM_CUDA(cudaMemcpyAsync(s_tids.p + coff[j], d_tids + pool->h_off[i], (coff[j + 1] - coff[j]) * 4ull,
                                        cudaMemcpyDeviceToDevice, st));
            }
            batmap_set S;
            S.params = P;
            S.params.tile = 0;
            S.m = m;
            S.n = cn;
            S.stream = st;
            S.skip_schedule = true;
            build_set(&S, s_off.p, s_tids.p, d_perm ? pool->d_perm.p : nullptr);
            pool->shift = S.shift;
            BM_CUDA(cudaMemcpyAsync(pool->d_bm.p + bm_pos, S.d_bm.p, S.bytes, cudaMemcpyDeviceToDevice, st));
            std::vector<uint64_t> cf(cn + 1, 0);
            BM_CUDA(cudaMemcpyAsync(cf.data(), S.d_fail_off.p, (cn + 1) * 8ull, cudaMemcpyDeviceToHost, st));
            BM_CUDA(cudaStreamSynchronize(st));
            if (S.n_failed) {
                std::vector<uint32_t> ft(S.n_failed);
                BM_CUDA(cudaMemcpy(ft.data(), S.d_fail_tid.p, S.n_failed * 4ull, cudaMemcpyDeviceToHost));
                f_chunks_tid.insert(f_chunks_tid.end(), ft.begin(), ft.end());
            }
            for (uint32_t j = 0; j < cn; j++) {
                base[c0 + j] = bm_pos + S.byte_off[S.rank[j]];
                uint32_t lg = 0;
                while ((1u << lg) < S.range[j]) lg++;
                rlog[c0 + j] = lg;
                f_off[c0 + j + 1] = f_pos + cf[j + 1];
            }
            f_pos += S.n_failed;
            bm_pos += S.bytes;
            pool->n_failed += S.n_failed;
            c0 = c1;
        }
        pool->bm_bytes = bm_pos;
        pool->d_fail_tid.alloc(std::max<uint64_t>(f_chunks_tid.size(), 1));
        if (!f_chunks_tid.empty())
            BM_CUDA(cudaMemcpyAsync(pool->d_fail_tid.p, f_chunks_tid.data(), f_chunks_tid.size() * 4ull,
                                    cudaMemcpyHostToDevice, st));
        BM_CUDA(cudaStreamSynchronize(st));
    }
    pool->d_fail_off.alloc(nb + 1);
    BM_CUDA(cudaMemcpyAsync(pool->d_fail_off.p, f_off.data(), (nb + 1) * 8ull, cudaMemcpyHostToDevice, st));
    pool->d_bm_base.alloc(std::max<uint32_t>(nb, 1));
    pool->d_bm_rlog.alloc(std::max<uint32_t>(nb, 1));
    if (nb) {
        BM_CUDA(cudaMemcpyAsync(pool->d_bm_base.p, base.data(), nb * 8ull, cudaMemcpyHostToDevice, st));
        BM_CUDA(cudaMemcpyAsync(pool->d_bm_rlog.p, rlog.data(), nb * 4ull, cudaMemcpyHostToDevice, st));
    }
    pool->view = PoolView{pool->d_off.p,     pool->d_tids.p,     make_perm_view(d_perm ? pool->d_perm.p : nullptr, m, P.perm_seed),
                          pool->d_bm_index.p, pool->d_bm_base.p, pool->d_bm_rlog.p,
                          pool->d_fail_off.p, pool->d_fail_tid.p, pool->d_bm.p,
                          m,                  nb ? pool->shift : shift,
                          pool->d_idx_off.p,  pool->d_idx.p};
    BM_CUDA(cudaStreamSynchronize(st));
    *out = pool.release();
}

// Up to so many tasks come from the host, more are made by a launch of k_query_tasks: 4 us, a fifth
// of the latency of a small batch.  A pool of 500 sets of 2 to 60: Poisson arrivals p50 23.3 -> 19.4 us;
// 3,000 queries at once, one by one 63.4 -> 53.2 ms, 16 a batch 2.44 -> 2.05, 256 a batch 0.217 -> 0.203
// (sets of 5 to 5,000, where the host sets the pace: 0.225 -> 0.235).
constexpr uint64_t HOST_TASKS = 256;

// A batch of queries on the host: descriptors with the smallest set first, and the
// first task of each (one more: the number of tasks), tasks of `elems` elements;
// the tasks themselves (the first tasks() of host_tasks) if there are at most HOST_TASKS.
struct Batch {
    std::vector<QueryDesc> qs;
    std::vector<uint32_t> size, first;
    std::vector<ProbeTask> host_tasks = std::vector<ProbeTask>(HOST_TASKS);
    uint32_t elems = 0;
    uint64_t tasks() const { return first.empty() ? 0 : first.back(); }
};

// elems 0: chosen by the work.
static void prepare_batch(const batmap_pool *pool, const uint32_t *qoff, const uint32_t *ids, uint64_t q0, uint64_t q1,
                          Batch &B, uint32_t elems) {
    B.qs.resize(q1 - q0);
    B.size.resize(q1 - q0);
    B.first.resize(q1 - q0 + 1);
    auto size_of = [&](uint32_t c) { return pool->h_off[c + 1] - pool->h_off[c]; };
    uint64_t total = 0;
    for (uint64_t q = q0; q < q1; q++) {
        const uint32_t k = qoff[q + 1] - qoff[q];
        BM_REQUIRE(k >= 1 && k <= MAX_K, BATMAP_ERR_ARG, "each query names 1..8 sets");
        QueryDesc &d = B.qs[q - q0];
        d.k = k;
        for (uint32_t t = 0; t < k; t++) {
            const uint32_t c = ids[qoff[q] + t];
            BM_REQUIRE(c < pool->n, BATMAP_ERR_ARG, "query names a set id >= n");
            d.ids[t] = c;
        }
        std::sort(d.ids, d.ids + k, [&](uint32_t a, uint32_t b) {
            const uint64_t sa = size_of(a), sb = size_of(b);
            return sa < sb || (sa == sb && a < b);
        });
        B.size[q - q0] = (uint32_t)size_of(d.ids[0]);  // <= 2^30
        total += B.size[q - q0];
    }
    // Small batches: shorter tasks until there are some for every warp that the chip holds.
    if (!elems)
        for (elems = TASK_ELEMS; elems > 128 && total / elems < 8192;) elems /= 2;
    B.elems = elems;
    uint64_t nt = 0;
    for (uint64_t q = 0; q < q1 - q0; q++) {
        B.first[q] = (uint32_t)nt;
        nt += (B.size[q] + elems - 1) / elems;
    }
    BM_REQUIRE(nt < (1ull << 32), BATMAP_ERR_ARG, "too much work in one call");
    B.first[q1 - q0] = (uint32_t)nt;
    if (nt > HOST_TASKS) return;
    for (uint64_t q = 0; q < q1 - q0; q++)
        for (uint32_t t = B.first[q], at = 0; t < B.first[q + 1]; t++, at += elems)
            B.host_tasks[t] = {(uint32_t)q, at, std::min(B.size[q], at + elems)};
}

static unsigned probe_blocks(uint64_t tasks) { return (unsigned)((tasks + PROBE_WARPS - 1) / PROBE_WARPS); }

static uint64_t query_work(const batmap_pool *pool, const uint32_t *qoff, const uint32_t *ids, uint64_t q) {
    uint64_t small = UINT64_MAX;
    for (uint32_t t = qoff[q]; t < qoff[q + 1]; t++) {
        const uint32_t c = ids[t];
        if (c < pool->n) small = std::min<uint64_t>(small, pool->h_off[c + 1] - pool->h_off[c]);
    }
    return (small == UINT64_MAX ? 0 : small) * (qoff[q + 1] - qoff[q]) + 1;
}

// The descriptors and tasks of a batch on the device, copied from the host's arrays (qs, first,
// and tasks or, where there are many, nullptr).
static void upload_batch(const batmap_pool *pool, const QueryDesc *qs, uint64_t nq, QueryDesc *d_q, const uint32_t *first,
                         uint32_t *d_first, uint32_t elems, const ProbeTask *tasks, ProbeTask *d_t, cudaStream_t st) {
    const uint64_t nt = first[nq];
    if (!nt) return;
    if (tasks) BM_CUDA(cudaMemcpyAsync(d_t, tasks, nt * sizeof(ProbeTask), cudaMemcpyHostToDevice, st));
    else BM_CUDA(cudaMemcpyAsync(d_first, first, (nq + 1) * sizeof(uint32_t), cudaMemcpyHostToDevice, st));
    BM_CUDA(cudaMemcpyAsync(d_q, qs, nq * sizeof(QueryDesc), cudaMemcpyHostToDevice, st));
    if (tasks) return;
    k_query_tasks<<<(unsigned)nq, 64, 0, st>>>(pool->view.off, d_q, d_first, elems, d_t);
    BM_CHECK_LAUNCH();
}

// Answers as element lists: out_off[q] .. out_off[q+1] in out (ascending).
static void intersect_list(const batmap_pool *pool, const uint32_t *qoff, const uint32_t *ids, uint32_t nq,
                           uint64_t *d_out_off, uint32_t *d_out, uint64_t cap, uint64_t *n_total, cudaStream_t st) {
    BM_REQUIRE(pool && qoff && n_total && d_out_off, BATMAP_ERR_ARG, "NULL argument");
    BM_REQUIRE(cap == 0 || d_out, BATMAP_ERR_ARG, "d_out is NULL with cap > 0");
    Workspace ws(st);
    Batch B;
    prepare_batch(pool, qoff, ids, 0, nq, B, 0);
    const uint64_t nt = B.tasks();
    WsBuf<QueryDesc> d_q(ws, std::max<uint64_t>(nq, 1));
    WsBuf<ProbeTask> d_t(ws, std::max<uint64_t>(nt, 1));
    WsBuf<uint64_t> d_toff(ws, nt + 1), d_total(ws, 1);
    WsBuf<uint32_t> d_first(ws, nq + 1);
    const ProbeTask *host = nt <= HOST_TASKS ? B.host_tasks.data() : nullptr;
    upload_batch(pool, B.qs.data(), nq, d_q.p, B.first.data(), d_first.p, B.elems, host, d_t.p, st);
    if (host || !nt)  // (else it is there)
        BM_CUDA(cudaMemcpyAsync(d_first.p, B.first.data(), (nq + 1ull) * sizeof(uint32_t), cudaMemcpyHostToDevice, st));
    WsBuf<uint32_t> d_masks(ws, cap ? 32 * nt : 0);
    if (nt) {
        k_probe<<<probe_blocks(nt), 32 * PROBE_WARPS, 0, st>>>(pool->view, d_q.p, d_t.p, (uint32_t)nt, nullptr, d_toff.p,
                                                               cap ? d_masks.p : nullptr);
        BM_CHECK_LAUNCH();
    }
    WsBuf<uint64_t> scan_state(ws, scan_states(nt));
    scan_with_tail(d_toff.p, nt, d_total.p, scan_state.p, st);
    k_query_offsets<<<(nq + 1 + 255) / 256, 256, 0, st>>>(d_toff.p, d_first.p, nq, d_out_off);
    BM_CHECK_LAUNCH();
    if (nt && cap) {
        k_probe_write<<<(unsigned)((nt + 7) / 8), 256, 0, st>>>(pool->view, d_q.p, d_t.p, (uint32_t)nt, d_toff.p, d_masks.p,
                                                                d_out, cap);
        BM_CHECK_LAUNCH();
    }
    uint64_t total = 0;
    BM_CUDA(cudaMemcpyAsync(&total, d_total.p, 8, cudaMemcpyDeviceToHost, st));
    BM_CUDA(cudaStreamSynchronize(st));
    ws.done();
    check_total(total);
    *n_total = total;
    if (total > cap)
        throw Error{BATMAP_ERR_CAPACITY, "d_out too small: " + std::to_string(total) + " elements in the answers"};
}

// Staging for one in-flight batch (pinned host + device, fixed capacity).
struct Slot {
    cudaStream_t st = nullptr;
    cudaEvent_t done = nullptr;
    QueryDesc *h_q = nullptr;
    uint32_t *h_first = nullptr;
    ProbeTask *h_t = nullptr;  // [HOST_TASKS]
    DevBuf<QueryDesc> d_q;
    DevBuf<uint32_t> d_first;
    DevBuf<ProbeTask> d_t;
    uint64_t qcap = 0, tcap = 0;
    uint64_t q0 = 0, q1 = 0, work = 0;
    bool busy = false;
    void init(uint64_t qc, uint64_t tc) {
        qcap = qc;
        tcap = tc;
        BM_CUDA(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
        BM_CUDA(cudaEventCreateWithFlags(&done, cudaEventDisableTiming));
        BM_CUDA(cudaMallocHost(&h_q, qc * sizeof(QueryDesc)));
        BM_CUDA(cudaMallocHost(&h_first, (qc + 1) * sizeof(uint32_t)));
        BM_CUDA(cudaMallocHost(&h_t, HOST_TASKS * sizeof(ProbeTask)));
        d_q.alloc(qc);
        d_first.alloc(qc + 1);
        d_t.alloc(tc);
    }
    void destroy() {
        if (done) cudaEventDestroy(done);
        if (st) cudaStreamDestroy(st);
        if (h_q) cudaFreeHost(h_q);
        if (h_first) cudaFreeHost(h_first);
        if (h_t) cudaFreeHost(h_t);
        done = nullptr;
        st = nullptr;
        h_q = nullptr;
        h_first = nullptr;
        h_t = nullptr;
    }
};

// Uploads a batch and counts its answers (zeroed first).
static void launch_probe(const batmap_pool *pool, const QueryDesc *qs, uint64_t nq, QueryDesc *d_q, const uint32_t *first,
                         uint32_t *d_first, uint32_t elems, const ProbeTask *tasks, ProbeTask *d_t,
                         unsigned long long *d_counts, cudaStream_t st) {
    const uint64_t nt = first[nq];
    upload_batch(pool, qs, nq, d_q, first, d_first, elems, tasks, d_t, st);
    BM_CUDA(cudaMemsetAsync(d_counts, 0, nq * sizeof(unsigned long long), st));
    if (nt) {
        k_probe<<<probe_blocks(nt), 32 * PROBE_WARPS, 0, st>>>(pool->view, d_q, d_t, (uint32_t)nt, d_counts, nullptr, nullptr);
        BM_CHECK_LAUNCH();
    }
}

static void launch_batch(const batmap_pool *pool, Slot &S, const Batch &B, unsigned long long *d_counts) {
    std::memcpy(S.h_q, B.qs.data(), B.qs.size() * sizeof(QueryDesc));
    std::memcpy(S.h_first, B.first.data(), B.first.size() * sizeof(uint32_t));
    if (B.tasks() <= HOST_TASKS) std::memcpy(S.h_t, B.host_tasks.data(), B.tasks() * sizeof(ProbeTask));
    launch_probe(pool, S.h_q, B.qs.size(), S.d_q.p, S.h_first, S.d_first.p, B.elems,
                 B.tasks() <= HOST_TASKS ? S.h_t : nullptr, S.d_t.p, d_counts + S.q0, S.st);
    BM_CUDA(cudaEventRecord(S.done, S.st));
}

static void intersect(const batmap_pool *pool, const uint32_t *qoff, const uint32_t *ids, uint32_t nq,
                      unsigned long long *d_counts, cudaStream_t st) {
    BM_REQUIRE(pool && qoff && (nq == 0 || ids) && (nq == 0 || d_counts), BATMAP_ERR_ARG, "NULL argument");
    if (!nq) return;
    Batch B;
    prepare_batch(pool, qoff, ids, 0, nq, B, 0);
    Workspace ws(st);
    WsBuf<QueryDesc> d_q(ws, nq);
    WsBuf<uint32_t> d_first(ws, nq + 1);
    WsBuf<ProbeTask> d_t(ws, B.tasks());
    launch_probe(pool, B.qs.data(), nq, d_q.p, B.first.data(), d_first.p, B.elems,
                 B.tasks() <= HOST_TASKS ? B.host_tasks.data() : nullptr, d_t.p, d_counts, st);
    BM_CUDA(cudaStreamSynchronize(st));
    ws.done();
}

// The continuous-batching request loop.  Queries arrive at h_arrival[q]
// seconds after the start (non-decreasing).  Whenever a slot is free, the
// loop gathers the queries that have arrived and not been submitted, up to
// max_batch queries and while the work in flight stays within the budget
// (work = elements of the smallest set x sets named), copies their
// descriptors to the slot's device buffers and launches them on the slot's
// stream; batches on different slots overlap on the device.  A query's
// latency is the host time at which its batch's completion event was
// observed minus its arrival time.
static void serve(const batmap_pool *pool, const uint32_t *qoff, const uint32_t *ids, const double *arrival,
                  uint32_t nq, const batmap_serve_opts *o, uint64_t *h_counts, double *h_latency,
                  batmap_serve_stats *stats, cudaStream_t st) {
    BM_REQUIRE(pool && qoff && arrival && h_counts && h_latency, BATMAP_ERR_ARG, "NULL argument");
    batmap_serve_opts opt{64, 4, 1ull << 26, 0};
    if (o) opt = *o;
    BM_REQUIRE(opt.max_batch >= 1 && opt.slots >= 1 && opt.slots <= 64, BATMAP_ERR_ARG, "bad serve options");
    for (uint32_t q = 1; q < nq; q++)
        BM_REQUIRE(arrival[q] >= arrival[q - 1], BATMAP_ERR_ARG, "arrival times must be non-decreasing");
    std::vector<uint64_t> work(nq);
    uint64_t max_tasks = 1, max_work = 1;
    for (uint32_t q = 0; q < nq; q++) {
        work[q] = query_work(pool, qoff, ids, q);
        max_work = std::max(max_work, work[q]);
    }
    // task capacity of a slot: the largest batch the budget admits
    for (uint32_t q = 0; q < nq; q++) {
        uint64_t small = work[q] / std::max<uint32_t>(1, qoff[q + 1] - qoff[q]);
        max_tasks = std::max<uint64_t>(max_tasks, small / TASK_ELEMS + 1);
    }
    const uint64_t budget = std::max<uint64_t>(opt.work_budget, max_work);
    const uint64_t tcap = std::max<uint64_t>(max_tasks * 2, budget / TASK_ELEMS + (uint64_t)opt.max_batch);
    DevBuf<unsigned long long> d_counts(std::max<uint32_t>(nq, 1));
    std::vector<Slot> slots(opt.slots);
    for (auto &s : slots) s.init(opt.max_batch, tcap);
    Batch B;
    using clk = std::chrono::steady_clock;
    const auto t0 = clk::now();
    auto now_s = [&] { return std::chrono::duration<double>(clk::now() - t0).count(); };
    uint64_t next = 0, done = 0, inflight_work = 0, batches = 0, max_inflight = 0, inflight = 0;
    try {
        while (done < nq) {
            const double t = now_s();
            bool progressed = false;
            for (auto &s : slots) {
                if (!s.busy) continue;
                cudaError_t e = cudaEventQuery(s.done);
                if (e == cudaErrorNotReady) continue;
                BM_CUDA(e);
                const double tc = now_s();
                for (uint64_t q = s.q0; q < s.q1; q++) h_latency[q] = tc - arrival[q];
                done += s.q1 - s.q0;
                inflight_work -= s.work;
                inflight--;
                s.busy = false;
                progressed = true;
            }
            for (auto &s : slots) {
                if (s.busy || next >= nq || arrival[next] > t) continue;
                uint64_t q1 = next, w = 0;
                while (q1 < nq && arrival[q1] <= t && q1 - next < opt.max_batch &&
                       (q1 == next ? inflight_work + work[q1] <= budget || inflight == 0
                                   : inflight_work + w + work[q1] <= budget))
                    w += work[q1++];
                if (q1 == next) break;  // budget full: wait for completions
                prepare_batch(pool, qoff, ids, next, q1, B, TASK_ELEMS);
                if (B.tasks() > s.tcap) {  // admit fewer queries
                    q1 = next + 1;
                    prepare_batch(pool, qoff, ids, next, q1, B, TASK_ELEMS);
                    BM_REQUIRE(B.tasks() <= s.tcap, BATMAP_ERR_INTERNAL, "task capacity");
                    w = work[next];
                }
                s.q0 = next;
                s.q1 = q1;
                s.work = w;
                launch_batch(pool, s, B, d_counts.p);
                s.busy = true;
                inflight++;
                inflight_work += w;
                max_inflight = std::max(max_inflight, inflight);
                batches++;
                next = q1;
                progressed = true;
            }
            if (!progressed) {
                const double wait = next < nq ? arrival[next] - now_s() : 0.0;
                if (wait > 200e-6) std::this_thread::sleep_for(std::chrono::microseconds(50));
            }
        }
        const double makespan = now_s();
        if (nq) BM_CUDA(cudaMemcpy(h_counts, d_counts.p, nq * sizeof(uint64_t), cudaMemcpyDeviceToHost));
        if (stats) {
            std::memset(stats, 0, sizeof(*stats));
            stats->makespan_s = makespan;
            stats->batches = batches;
            stats->max_inflight = max_inflight;
            std::vector<double> lat(h_latency, h_latency + nq);
            std::sort(lat.begin(), lat.end());
            if (nq) {
                stats->p50_s = lat[(size_t)(0.50 * (nq - 1))];
                stats->p99_s = lat[(size_t)(0.99 * (nq - 1))];
                stats->max_s = lat.back();
                stats->queries_per_s = nq / std::max(makespan, 1e-9);
            }
        }
    } catch (...) {
        for (auto &s : slots) {
            if (s.st) cudaStreamSynchronize(s.st);
            s.destroy();
        }
        throw;
    }
    for (auto &s : slots) {
        cudaStreamSynchronize(s.st);
        s.destroy();
    }
}

}  // namespace bm

extern "C" {

#define BM_GUARD(body)                              \
    try {                                           \
        body;                                       \
        return BATMAP_OK;                           \
    } catch (const bm::Error &e) {                  \
        bm::set_error(e.msg);                       \
        return e.code;                              \
    } catch (...) {                                 \
        bm::set_error("unexpected internal error"); \
        return BATMAP_ERR_INTERNAL;                 \
    }

batmap_status batmap_pool_create(const batmap_params *p, uint32_t m, uint32_t n, const uint64_t *d_offsets,
                                 const uint32_t *d_tids, const uint32_t *d_perm, cudaStream_t stream,
                                 batmap_pool **out) {
    BM_GUARD(bm::pool_create(p, m, n, d_offsets, d_tids, d_perm, stream, out));
}

void batmap_pool_free(batmap_pool *pool) { delete pool; }

batmap_status batmap_pool_info(const batmap_pool *pool, uint32_t *n_batmaps, uint64_t *batmap_bytes,
                               uint64_t *n_elements) {
    BM_GUARD({
        BM_REQUIRE(pool, BATMAP_ERR_ARG, "NULL pool");
        if (n_batmaps) *n_batmaps = pool->n_big;
        if (batmap_bytes) *batmap_bytes = pool->bm_bytes;
        if (n_elements) *n_elements = pool->h_off[pool->n];
    });
}

batmap_status intersect_query(const batmap_pool *pool, const uint32_t *h_qoff, const uint32_t *h_ids,
                              uint32_t n_queries, uint64_t *d_counts, cudaStream_t stream) {
    BM_GUARD(bm::intersect(pool, h_qoff, h_ids, n_queries, reinterpret_cast<unsigned long long *>(d_counts),
                           stream));
}

batmap_status intersect_query_list(const batmap_pool *pool, const uint32_t *h_qoff, const uint32_t *h_ids,
                                   uint32_t n_queries, uint64_t *d_out_off, uint32_t *d_out, uint64_t cap,
                                   uint64_t *n_total, cudaStream_t stream) {
    BM_GUARD(bm::intersect_list(pool, h_qoff, h_ids, n_queries, d_out_off, d_out, cap, n_total, stream));
}

batmap_status batmap_serve(const batmap_pool *pool, const uint32_t *h_qoff, const uint32_t *h_ids,
                           const double *h_arrival_s, uint32_t n_queries, const batmap_serve_opts *opts,
                           uint64_t *h_counts, double *h_latency_s, batmap_serve_stats *stats, cudaStream_t stream) {
    BM_GUARD(bm::serve(pool, h_qoff, h_ids, h_arrival_s, n_queries, opts, h_counts, h_latency_s, stats, stream));
}

}  // extern "C"

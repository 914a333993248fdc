// BatMap construction on the GPU (Sec. II and Sec. III-A/C).
//
//   validate  : tids strictly increasing and < m per item; each permutation
//               row a bijection of [0, m)
//   size      : s, r_0, r_i, widths 3 r_i, width-sorted order (host)
//   place     : parallel generalised cuckoo INSERT; every element with exactly
//               two copies gets its two bytes (indicator << 7 | code); the
//               rest are failed insertions (place.cu)
//   failures  : F_i in (item, tid) order, then the correction entries: one
//               (min, max) item pair per failed common transaction
//   schedule  : compare work units (host, compare.cu)
#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>
#include <numeric>

#include "bits.cuh"
#include "common.cuh"
#include "items.cuh"
#include "perm.cuh"
#include "place.cuh"
#include "scan.cuh"

namespace bm {

void build_schedule(batmap_set *S);  // compare.cu

// ---- validation ---------------------------------------------------------------

__global__ void k_validate_tids(ItemView v, uint32_t m, int *err) {
    uint32_t item;
    uint64_t e0, e1;
    chunk_range(v, blockIdx.x, &item, &e0, &e1);
    for (uint64_t e = e0 + threadIdx.x; e < e1; e += TPB) {
        uint32_t x = v.tids[e];
        bool bad = x >= m;
        if (e + 1 < v.off[item + 1]) bad |= !(x < v.tids[e + 1]);
        if (bad) atomicExch(err, 1);
    }
}

__global__ void k_validate_perm(const uint32_t *perm, uint32_t m, uint32_t rows, uint32_t *bits, int *err) {
    uint64_t total = (uint64_t)rows * m;
    for (uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; q < total;
         q += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t t = (uint32_t)(q / m);
        uint32_t val = perm[q];
        if (val >= m) {
            atomicExch(err, 2);
            continue;
        }
        uint64_t w = (uint64_t)t * ((m + 31) / 32) + val / 32;
        uint32_t bit = 1u << (val % 32);
        uint32_t old = atomicOr(&bits[w], bit);
        if (old & bit) atomicExch(err, 2);
    }
}

// Chunk b: elements [ch_start[b], + CHUNK) of item ch_item[b].
__global__ void k_chunks(const uint64_t *off, const uint32_t *chunk0, uint32_t *ch_item, uint64_t *ch_start) {
    const uint32_t i = blockIdx.x;
    const uint64_t e0 = off[i], e1 = off[i + 1];
    for (uint64_t c = threadIdx.x; e0 + c * CHUNK < e1; c += blockDim.x) {
        ch_item[chunk0[i] + c] = i;
        ch_start[chunk0[i] + c] = e0 + c * CHUNK;
    }
}

// Number of correction entries of a set with bit rows, which needs no list of
// them: a failed (a, x) makes one with every other item holding x, less one per
// pair of items that both failed x.  One warp per failure counts the items in
// x's column; seen: m zeroed words.
__global__ void k_count_corrections(const uint32_t *f_tid, uint64_t nfail, const uint8_t *bits, uint32_t n,
                                    uint32_t *seen, unsigned long long *count) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x / 32);
    for (uint64_t k = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) / 32; k < nfail; k += warps) {
        const uint32_t x = f_tid[k];
        const uint8_t *col = bits + (uint64_t)(x >> 8) * 32u * n + 4u * ((x >> 5) & 7u);
        uint32_t items = 0;
        for (uint32_t c = lane; c < n; c += 32)
            items += (*reinterpret_cast<const uint32_t *>(col + 32ull * c) >> (x & 31u)) & 1u;
        items = __reduce_add_sync(0xffffffffu, items);
        if (lane == 0) atomicAdd(count, (unsigned long long)items - 1ull - atomicAdd(&seen[x], 1u));
    }
}

// ---- failed insertions ------------------------------------------------------------

// f_off[i] = first failure of item i (lower bound in the sorted f_item list).
__global__ void k_fail_offsets(const uint32_t *f_item, uint64_t nfail, uint32_t n, uint64_t *f_off) {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i > n) return;
    uint64_t lo = 0, hi = nfail;
    while (lo < hi) {
        uint64_t mid = (lo + hi) >> 1;
        if (f_item[mid] < i) lo = mid + 1; else hi = mid;
    }
    f_off[i] = lo;
}

// ---- correction entries (Sec. III-C "Failed insertions") --------------------------
//
// For a failed (a, x) and every item c != a containing x, the pair {a, c}
// misses x in the BatMap comparison.  When x failed in c as well, the pair
// is generated from the smaller id only, so each (x, pair) is added once.

__global__ void k_mark_failed(const uint32_t *f_tid, uint64_t nfail, uint32_t *bits) {
    for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < nfail;
         k += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t x = f_tid[k];
        atomicOr(&bits[x >> 5], 1u << (x & 31));
    }
}

__global__ void k_popc_words(const uint32_t *bits, uint64_t nwords, uint64_t *out) {
    for (uint64_t w = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; w < nwords;
         w += (uint64_t)gridDim.x * blockDim.x)
        out[w] = __popc(bits[w]);
}

__device__ __forceinline__ bool failed_bit(const uint32_t *bits, uint32_t x) {
    return (bits[x >> 5] >> (x & 31)) & 1u;
}

__device__ __forceinline__ uint32_t bit_rank(const uint32_t *bits, const uint64_t *wrank, uint32_t x) {
    return (uint32_t)(wrank[x >> 5] + __popc(bits[x >> 5] & ((1u << (x & 31)) - 1u)));
}

__global__ void k_count_per_tid(const uint32_t *f_tid, uint64_t nfail, const uint32_t *bits,
                                const uint64_t *wrank, uint64_t *cnt) {
    for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < nfail;
         k += (uint64_t)gridDim.x * blockDim.x)
        atomicAdd((unsigned long long *)&cnt[bit_rank(bits, wrank, f_tid[k])], 1ull);
}

__global__ void k_fill_per_tid(const uint32_t *f_item, const uint32_t *f_tid, uint64_t nfail,
                               const uint32_t *bits, const uint64_t *wrank, const uint64_t *fptr,
                               unsigned long long *cursor, uint32_t *fitems) {
    for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < nfail;
         k += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t u = bit_rank(bits, wrank, f_tid[k]);
        uint64_t p = fptr[u] + atomicAdd(&cursor[u], 1ull);
        fitems[p] = f_item[k];
    }
}

template <bool WRITE>
__global__ void k_corrections(ItemView v, uint32_t m, const uint32_t *bits, const uint64_t *wrank,
                              const uint64_t *fptr, const uint32_t *fitems,
                              unsigned long long *counter, uint32_t *corr) {
    uint32_t c;
    uint64_t e0, e1;
    chunk_range(v, blockIdx.x, &c, &e0, &e1);
    for (uint64_t e = e0 + threadIdx.x; e < e1; e += TPB) {
        uint32_t x = v.tids[e];
        if (x >= m || !failed_bit(bits, x)) continue;
        uint32_t u = bit_rank(bits, wrank, x);
        uint64_t b0 = fptr[u], b1 = fptr[u + 1];
        bool c_failed = false;
        for (uint64_t k = b0; k < b1; k++) c_failed |= (fitems[k] == c);
        for (uint64_t k = b0; k < b1; k++) {
            uint32_t a = fitems[k];
            if (a == c) continue;
            if (c_failed && c < a) continue;  // generated from c's side
            unsigned long long slot = atomicAdd(counter, 1ull);
            if (WRITE) {
                corr[2 * slot] = a < c ? a : c;
                corr[2 * slot + 1] = a < c ? c : a;
            }
        }
    }
}

// ---- host side -------------------------------------------------------------------

PermView make_perm_view(const uint32_t *table, uint32_t m, uint64_t seed) {
    PermView P{};
    P.table = table;
    P.m = m;
    uint32_t b = 0;
    while (b < 32 && (1ull << b) < (uint64_t)m) b++;  // ceil(log2 m)
    b = std::max<uint32_t>(b, 2);
    b += b & 1u;
    P.half = b / 2;
    P.mask = (1u << P.half) - 1u;
    // SplitMix64 from the seed: four round keys per table, low 32 bits each
    uint64_t state = seed;
    uint32_t k[4 * PERM_MAX_TABLES];
    for (int j = 0; j < 4 * PERM_MAX_TABLES; j++) {
        state += 0x9E3779B97F4A7C15ull;
        uint64_t z = state;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        k[j] = (uint32_t)(z ^ (z >> 31));
    }
    for (int t = 0; t < PERM_MAX_TABLES; t++) P.key[t] = make_uint4(k[4 * t], k[4 * t + 1], k[4 * t + 2], k[4 * t + 3]);
    return P;
}

static uint32_t shift_bits(uint32_t m, uint32_t min_shift) {
    uint32_t s = min_shift;
    while ((uint64_t)m > 127ull << s) s++;
    return s;
}

// The placement scratch (the regions of place.cu: 96 MiB, 184 for 3-of-4 and
// 4-of-5 sets of wide items, or two of the widest item's tables if that is more;
// and 8 bytes per 2,048 slots and per 1,024 elements of the items placed there, 61 MiB
// at m = 2^22, n = 8,192, 5%) is kept between builds so that repeated builds do not
// pay for allocating and freeing it; it is released when a build needs less than a
// quarter of it or on batmap_release_scratch().  Builds are serialised on it.
std::mutex g_scratch_mu;
static DevBuf<uint32_t> g_scratch;

DevBuf<uint32_t> &scratch_table(uint64_t slots) {
    if (g_scratch.n < slots || g_scratch.n > 4 * slots + (1u << 20)) g_scratch.alloc(slots);
    return g_scratch;
}

void release_scratch() {
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    g_scratch.release();
    bm_buffer_release_all();
    release_arenas();
}

// ---- kept device memory and events ---------------------------------------------------

namespace {
struct CachedBuf {
    uint8_t *p;
    size_t cap;
};
std::mutex g_bm_cache_mu;
std::vector<CachedBuf> g_bm_cache[2];  // arrays of up to LARGE_BUF bytes, larger ones; oldest first
constexpr size_t LARGE_BUF = 64ull << 20, BM_CACHE[2] = {32, 4};
thread_local int t_released = 0;

std::mutex g_event_mu;
std::vector<cudaEvent_t> g_events;  // at most MAX_EVENTS
constexpr size_t MAX_EVENTS = 256;
}  // namespace

// ---- device memory ----

namespace {
std::atomic<uint64_t> g_device_bytes{0}, g_device_limit{UINT64_MAX};
bool release_idle();
}  // namespace

void *device_alloc(size_t bytes) {
    for (bool again = false;; again = true) {
        void *p = nullptr;
        const cudaError_t e = g_device_bytes + bytes > g_device_limit ? cudaErrorMemoryAllocation : cudaMalloc(&p, bytes);
        if (e == cudaSuccess) {
            g_device_bytes += bytes;
            return p;
        }
        cudaGetLastError();  // reported here, not by the next launch's check
        BM_REQUIRE(e == cudaErrorMemoryAllocation, BATMAP_ERR_CUDA, std::string("cudaMalloc: ") + cudaGetErrorString(e));
        BM_REQUIRE(!again && release_idle(), BATMAP_ERR_NOMEM, "no device memory for " + std::to_string(bytes) + " bytes");
    }
}

void device_free(void *p, size_t bytes) {
    cudaFree(p);
    g_device_bytes -= bytes;
}

void set_memory_limit(uint64_t bytes) { g_device_limit = bytes ? g_device_bytes + bytes : UINT64_MAX; }

// Bytes of freed sets' arrays kept in all: a quarter of the device's memory.
static uint64_t kept_bytes() {
    static const uint64_t total = [] {
        size_t f = 0, t = 0;
        if (cudaMemGetInfo(&f, &t) != cudaSuccess) cudaGetLastError();
        return (uint64_t)t;
    }();
    return std::min<uint64_t>(total, g_device_limit) / 4;
}

uint8_t *bm_buffer_take(size_t bytes, size_t *capacity) {
    {
        std::lock_guard<std::mutex> lock(g_bm_cache_mu);
        CachedBuf *best = nullptr;
        std::vector<CachedBuf> *from = nullptr;
        for (auto &cache : g_bm_cache)
            for (auto &b : cache)
                if (b.cap >= bytes && b.cap <= 2 * bytes + (1u << 20) && (!best || b.cap < best->cap)) {
                    best = &b;
                    from = &cache;
                }
        if (best) {
            const CachedBuf b = *best;
            from->erase(from->begin() + (best - from->data()));
            *capacity = b.cap;
            return b.p;
        }
    }
    *capacity = bytes;
    return static_cast<uint8_t *>(device_alloc(bytes));
}

void bm_buffer_give(uint8_t *p, size_t capacity) {
    // no queued work may still use the array when it is handed out again
    if (!t_released) cudaDeviceSynchronize();
    std::lock_guard<std::mutex> lock(g_bm_cache_mu);
    const uint64_t most = kept_bytes();
    if (capacity > most) return device_free(p, capacity);
    const int k = capacity > LARGE_BUF;
    g_bm_cache[k].push_back({p, capacity});
    uint64_t held = 0;
    for (auto &cache : g_bm_cache)
        for (auto &b : cache) held += b.cap;
    for (;;) {
        // the oldest of its class, or of the large ones
        const int from = g_bm_cache[k].size() > BM_CACHE[k] ? k : held > most ? !g_bm_cache[1].empty() : -1;
        if (from < 0) break;
        const CachedBuf b = g_bm_cache[from].front();
        g_bm_cache[from].erase(g_bm_cache[from].begin());
        held -= b.cap;
        device_free(b.p, b.cap);
    }
}

void bm_buffer_release_all() {
    std::lock_guard<std::mutex> lock(g_bm_cache_mu);
    for (auto &cache : g_bm_cache) {
        for (auto &b : cache) device_free(b.p, b.cap);
        cache.clear();
    }
}

ReleaseScope::ReleaseScope() {
    cudaDeviceSynchronize();
    t_released++;
}
ReleaseScope::~ReleaseScope() { t_released--; }

void PhaseEvents::create() {
    if (ok) return;
    std::lock_guard<std::mutex> lock(g_event_mu);
    for (int i = 0; i < N; i++) {
        if (!g_events.empty()) {
            ev[i] = g_events.back();
            g_events.pop_back();
        } else {
            BM_CUDA(cudaEventCreate(&ev[i]));
        }
    }
    ok = true;
}

PhaseEvents::~PhaseEvents() {
    std::lock_guard<std::mutex> lock(g_event_mu);
    for (int i = 0; i < N; i++) {
        if (!ev[i]) continue;
        if (g_events.size() < MAX_EVENTS) g_events.push_back(ev[i]);
        else cudaEventDestroy(ev[i]);
    }
}

struct Arena {
    struct Block {
        uint8_t *p;
        size_t cap, used;
    };
    std::vector<Block> blocks;
    void *pinned = nullptr;
    size_t total() const {
        size_t t = 0;
        for (const Block &b : blocks) t += b.cap;
        return t;
    }
    void add(size_t cap) {
        blocks.push_back({static_cast<uint8_t *>(device_alloc(cap)), cap, 0});
    }
    void clear() {
        for (const Block &b : blocks) device_free(b.p, b.cap);
        blocks.clear();
    }
    ~Arena() {
        clear();
        if (pinned) cudaFreeHost(pinned);
    }
};

namespace {
std::mutex g_arena_mu;
std::vector<Arena *> g_arenas;
constexpr size_t MAX_ARENAS = 4, ARENA_BYTES = 256ull << 20;
}  // namespace

Workspace::Workspace(cudaStream_t st) : arena_(nullptr), st_(st) {
    std::lock_guard<std::mutex> lock(g_arena_mu);
    if (!g_arenas.empty()) {
        arena_ = g_arenas.back();
        g_arenas.pop_back();
    } else {
        arena_ = new Arena();
    }
}

Workspace::~Workspace() {
    if (!synced_) cudaStreamSynchronize(st_);
    // what took several blocks gets one next time
    const size_t total = arena_->total();
    try {
        if (arena_->blocks.size() > 1 || total > ARENA_BYTES) {
            arena_->clear();
            if (total <= ARENA_BYTES) arena_->add(total);
        }
    } catch (const Error &) {  // no memory to keep: the next call allocates what it needs
    }
    for (auto &b : arena_->blocks) b.used = 0;
    std::lock_guard<std::mutex> lock(g_arena_mu);
    if (g_arenas.size() < MAX_ARENAS) g_arenas.push_back(arena_);
    else delete arena_;
}

void *Workspace::bytes(size_t count) {
    if (!count) return nullptr;
    count = (count + 255) / 256 * 256;
    if (arena_->blocks.empty() || arena_->blocks.back().cap - arena_->blocks.back().used < count)
        arena_->add(std::max<size_t>(count, 1u << 20));
    Arena::Block &b = arena_->blocks.back();
    void *p = b.p + b.used;
    b.used += count;
    return p;
}

void *Workspace::host() {
    if (!arena_->pinned) BM_CUDA(cudaMallocHost(&arena_->pinned, PINNED));
    return arena_->pinned;
}

void release_arenas() {
    std::lock_guard<std::mutex> lock(g_arena_mu);
    for (Arena *a : g_arenas) delete a;
    g_arenas.clear();
}

namespace {
// Gives back the arrays and the scratch that no set and no call holds; false if there were none.
bool release_idle() {
    const uint64_t before = g_device_bytes;
    bm_buffer_release_all();
    release_arenas();
    return g_device_bytes != before;
}
}  // namespace

uint64_t device_available() {
    size_t free_b = 0, total_b = 0;
    BM_CUDA(cudaMemGetInfo(&free_b, &total_b));
    const uint64_t limit = g_device_limit, held = g_device_bytes;
    uint64_t b = std::min<uint64_t>(free_b, limit > held ? limit - held : 0) + g_scratch.bytes();
    {
        std::lock_guard<std::mutex> lock(g_bm_cache_mu);
        for (auto &cache : g_bm_cache)
            for (auto &c : cache) b += c.cap;
    }
    std::lock_guard<std::mutex> lock(g_arena_mu);
    for (const Arena *a : g_arenas) b += a->total();
    return b;
}

// ---- side stream ----

namespace {
cudaStream_t g_side = nullptr, g_more[SideStream::MORE];  // created at the first build, kept
cudaEvent_t g_fork = nullptr, g_join = nullptr;
}  // namespace

SideStream::SideStream(cudaStream_t st) : st_(st) {
    if (!g_side) {
        BM_CUDA(cudaEventCreateWithFlags(&g_fork, cudaEventDisableTiming));
        BM_CUDA(cudaEventCreateWithFlags(&g_join, cudaEventDisableTiming));
        for (cudaStream_t &s : g_more) BM_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
        BM_CUDA(cudaStreamCreateWithFlags(&g_side, cudaStreamNonBlocking));
    }
    side_ = g_side;
    BM_CUDA(cudaEventRecord(g_fork, st_));
    BM_CUDA(cudaStreamWaitEvent(side_, g_fork, 0));
}

cudaStream_t SideStream::more(uint32_t i) {
    BM_CUDA(cudaEventRecord(g_fork, st_));
    BM_CUDA(cudaStreamWaitEvent(g_more[i], g_fork, 0));
    used_ = i + 1;
    return g_more[i];
}

void SideStream::join() {
    if (joined_) return;
    BM_CUDA(cudaEventRecord(g_join, side_));
    BM_CUDA(cudaStreamWaitEvent(st_, g_join, 0));
    for (uint32_t i = 0; i < used_; i++) {
        BM_CUDA(cudaEventRecord(g_join, g_more[i]));
        BM_CUDA(cudaStreamWaitEvent(st_, g_join, 0));
    }
    joined_ = true;
}

SideStream::~SideStream() {
    if (joined_) return;  // an error on the way: nothing may outlive the call's memory
    cudaStreamSynchronize(side_);
    for (uint32_t i = 0; i < used_; i++) cudaStreamSynchronize(g_more[i]);
}

// The CSR offsets to the host (synchronises).
void read_offsets(Workspace &ws, std::vector<uint64_t> &off, const uint64_t *d_offsets, cudaStream_t st) {
    const size_t bytes = off.size() * sizeof(uint64_t);
    void *to = bytes <= Workspace::PINNED ? ws.host() : off.data();
    BM_CUDA(cudaMemcpyAsync(to, d_offsets, bytes, cudaMemcpyDeviceToHost, st));
    BM_CUDA(cudaStreamSynchronize(st));
    if (to != off.data()) std::memcpy(off.data(), to, bytes);
}

void build_set(batmap_set *S, const uint64_t *d_offsets, const uint32_t *d_tids,
               const uint32_t *d_perm) {
    std::lock_guard<std::mutex> scratch_lock(g_scratch_mu);
    const uint32_t m = S->m, n = S->n;
    cudaStream_t st = S->stream;
    Workspace ws(st);
    const batmap_params &P = S->params;
    PhaseEvents &E = S->build_ev;
    E.create();
    E.record(0, st);

    // CSR offsets on the host: sizes drive the layout and the schedule.
    std::vector<uint64_t> off(n + 1, 0);
    if (n) {
        BM_REQUIRE(d_offsets != nullptr, BATMAP_ERR_ARG, "d_offsets is NULL");
        read_offsets(ws, off, d_offsets, st);
    }
    BM_REQUIRE(off[0] == 0, BATMAP_ERR_ARG, "offsets[0] must be 0");
    for (uint32_t i = 0; i < n; i++)
        BM_REQUIRE(off[i + 1] >= off[i], BATMAP_ERR_ARG, "offsets must be non-decreasing");
    const uint64_t T = off[n];
    S->n_elements = T;
    BM_REQUIRE(T == 0 || d_tids != nullptr, BATMAP_ERR_ARG, "d_tids is NULL");
    const PermView PV = make_perm_view(d_perm, m, P.perm_seed);

    // ---- sizes (Sec. III-A) and width-sorted order (Sec. III-C) ----
    S->shift = shift_bits(m, P.min_shift);
    S->r0 = 1u << S->shift;
    std::vector<uint32_t> rlog(n);
    S->range.resize(n);
    for (uint32_t i = 0; i < n; i++) {
        rlog[i] = log2_range(off[i + 1] - off[i], P.load_num, P.load_den, S->shift);
        BM_REQUIRE(rlog[i] <= 31, BATMAP_ERR_ARG, "hash range exceeds 2^31");
        S->range[i] = 1u << rlog[i];
    }
    S->order.resize(n);
    // width-sorted (stable by id); in cross mode family A [0, n_a) first
    const uint32_t na = S->n_a;
    {
        uint32_t at[65] = {};
        auto key = [&](uint32_t i) { return rlog[i] + (na && i >= na ? 32u : 0u); };
        for (uint32_t i = 0; i < n; i++) at[key(i) + 1]++;
        for (int k = 0; k < 64; k++) at[k + 1] += at[k];
        for (uint32_t i = 0; i < n; i++) S->order[at[key(i)]++] = i;
    }
    S->rank.assign(n, 0);
    S->byte_off.assign(n, 0);
    S->wshift_sorted.assign(n, 0);
    // per-item arrays for the device: base (64 bits) | line_off | wshift | order | chunk0
    std::vector<uint32_t> meta(6ull * n);
    uint64_t *base = reinterpret_cast<uint64_t *>(meta.data());
    uint32_t *line_off = meta.data() + 2ull * n, *chunk0 = meta.data() + 5ull * n;
    uint64_t pos = 0;
    S->class_begin.clear();
    for (uint32_t q = 0; q < n; q++) {
        uint32_t i = S->order[q];
        S->rank[i] = q;
        S->byte_off[q] = pos;
        base[i] = pos;
        BM_REQUIRE(pos / 128 < (1ull << 32), BATMAP_ERR_ARG, "BatMap array exceeds 512 GB");
        line_off[q] = (uint32_t)(pos / 128);
        S->wshift_sorted[q] = rlog[i] - 2;
        if (q == 0 || rlog[S->order[q - 1]] != rlog[i] || (na && q == na)) S->class_begin.push_back(q);
        pos += 3ull << rlog[i];
    }
    S->class_begin.push_back(n);
    S->bytes = pos;
    // the compare kernel addresses BatMaps as 32-bit indices of 16-byte chunks
    BM_REQUIRE(pos <= (1ull << 36), BATMAP_ERR_ARG, "BatMaps of one set exceed 64 GB; split the instance");

    // algorithmic work of the compare: sum over pairs of the wider width / 4
    double wp = 0.0;
    if (!na) {
        for (uint32_t q = 0; q < n; q++) wp += (double)q * (double)((3ull << (S->wshift_sorted[q] + 2)) / 4);
    } else {
        // both families are width-sorted: A items no wider than b contribute b's width,
        // the wider ones their own (suffix sums over A)
        std::vector<double> suffix(na + 1, 0.0);
        for (uint32_t a = na; a-- > 0;) suffix[a] = suffix[a + 1] + (double)(3ull << S->wshift_sorted[a]);
        uint32_t a = 0;
        for (uint32_t b = na; b < n; b++) {
            while (a < na && S->wshift_sorted[a] <= S->wshift_sorted[b]) a++;
            wp += (double)a * (double)(3ull << S->wshift_sorted[b]) + suffix[a];
        }
    }
    S->word_pairs = wp;

    // ---- device metadata ----
    S->d_bm.alloc(S->bytes);
    uint32_t nch = 0;  // chunk b: CHUNK elements of one item
    for (uint32_t i = 0; i < n; i++) {
        chunk0[i] = nch;
        nch += (uint32_t)((off[i + 1] - off[i] + CHUNK - 1) / CHUNK);
    }
    if (n) {
        std::copy(S->wshift_sorted.begin(), S->wshift_sorted.end(), meta.begin() + 3ull * n);
        std::copy(S->order.begin(), S->order.end(), meta.begin() + 4ull * n);
        S->d_meta.alloc(meta.size());
        S->d_line_off.p = S->d_meta.p + 2ull * n;
        S->d_wshift.p = S->d_meta.p + 3ull * n;
        S->d_order.p = S->d_meta.p + 4ull * n;
        BM_CUDA(cudaMemcpyAsync(S->d_meta.p, meta.data(), meta.size() * 4, cudaMemcpyHostToDevice, st));
    }

    S->d_fail_off.alloc(n + 1);
    if (T == 0) {
        if (S->bytes) BM_CUDA(cudaMemsetAsync(S->d_bm.p, 0, S->bytes, st));
        BM_CUDA(cudaMemsetAsync(S->d_fail_off.p, 0, (n + 1) * sizeof(uint64_t), st));
        if (!S->skip_schedule) build_schedule(S);
        E.record(1, st);
        BM_CUDA(cudaStreamSynchronize(st));
        S->timing.build_ms = E.ms(0, 1);
        S->timing.place_ms = S->timing.finalize_ms = 0.f;
        return;
    }

    const uint64_t *d_base = reinterpret_cast<const uint64_t *>(S->d_meta.p);
    const uint32_t *d_chunk0 = S->d_meta.p + 5ull * n;
    WsBuf<uint32_t> d_ch_item(ws, nch);
    WsBuf<uint64_t> d_ch_start(ws, nch);
    ItemView v{d_offsets, d_tids, d_ch_item.p, d_ch_start.p};
    auto make_chunks = [&] {
        k_chunks<<<n, 64, 0, st>>>(d_offsets, d_chunk0, d_ch_item.p, d_ch_start.p);
        BM_CHECK_LAUNCH();
    };
    WsBuf<BuildStat> d_stat(ws, 1);
    BuildStat *stat = static_cast<BuildStat *>(ws.host());
    BM_CUDA(cudaMemsetAsync(d_stat.p, 0, sizeof(BuildStat), st));

    // ---- bit rows (where the pair supports come from them) and validation; the placement is safe on
    // lists and permutations that are refused behind it ----
    WsBuf<uint64_t> bs(ws, nch + 1);  // failed insertions per chunk
    WsBuf<uint32_t> d_mask(ws, (uint64_t)nch * (CHUNK / 32));
    BM_CUDA(cudaMemsetAsync(bs.p, 0, (nch + 1) * 8ull, st));
    const PermView place_perm = place_perms(PV, 3, off[n], ws, st);
    SideStream side(st);  // bit rows and the placement in shared memory, beside the placement in L2
    plan_contract(S, d_offsets, d_tids, d_stat.p->err + 2, P.validate != 0, side.side());
    if (P.validate && !S->contract) {  // (the bit rows' build checks every list)
        make_chunks();
        k_validate_tids<<<nch, TPB, 0, st>>>(v, m, d_stat.p->err);
        BM_CHECK_LAUNCH();
    }
    if (P.validate && d_perm) {  // computed permutations are bijections by construction
        WsBuf<uint32_t> d_bits(ws, 3ull * ((m + 31) / 32));
        BM_CUDA(cudaMemsetAsync(d_bits.p, 0, d_bits.bytes(), st));
        k_validate_perm<<<grid_for(3ull * m), 256, 0, st>>>(d_perm, m, 3, d_bits.p, d_stat.p->err);
        BM_CHECK_LAUNCH();
    }

    // ---- placement and bytes ----
    {
        E.record(2, st);
        std::vector<PlaceItem> list(n);
        for (uint32_t i = 0; i < n; i++) list[i] = {i, rlog[i], off[i + 1] - off[i]};
        WsBuf<uint32_t> d_list(ws, n), d_queue(ws, PLACE_QUEUES);
        PlaceJob J{};
        J.off = d_offsets;
        J.tids = d_tids;
        J.base = d_base;
        J.chunk0 = d_chunk0;
        J.shift = S->shift;
        J.max_moves = 3u * std::max<uint32_t>(P.max_loop, 1u);
        J.out = S->d_bm.p;
        J.fails = bs.p;
        J.mask = d_mask.p;
        J.queue = d_queue.p;
        J.refused = P.validate ? d_stat.p->err : nullptr;
        enqueue_place(3, J, place_perm, std::move(list), d_list.p, side);
        side.join();
        E.record(3, st);
        // failed insertions, ordered by (item, tid): counted and marked by the placement
        WsBuf<uint64_t> scan_state(ws, scan_states(nch));
        scan_with_tail(bs.p, nch, reinterpret_cast<uint64_t *>(&d_stat.p->nfail), scan_state.p, st);
        BM_CUDA(cudaMemsetAsync(S->d_fail_off.p, 0, (n + 1) * sizeof(uint64_t), st));
        if (!S->skip_schedule && !S->contract) build_schedule(S);
        E.record(4, st);
        E.record(1, st);
        BM_CUDA(cudaMemcpyAsync(stat, d_stat.p, sizeof(BuildStat), cudaMemcpyDeviceToHost, st));
        BM_CUDA(cudaStreamSynchronize(st));
        if (P.validate) stat->check();
        check_total(stat->nfail);
        const uint64_t nfail = stat->nfail;
        S->n_failed = nfail;
        WsBuf<uint32_t> f_item(ws, nfail);
        S->d_fail_tid.alloc(nfail);
        if (nfail) {
            make_chunks();
            k_failures<<<nch, TPB, 0, st>>>(v, d_mask.p, bs.p, f_item.p, S->d_fail_tid.p);
            BM_CHECK_LAUNCH();
            k_fail_offsets<<<(n + 1 + 255) / 256, 256, 0, st>>>(f_item.p, nfail, n, S->d_fail_off.p);
            BM_CHECK_LAUNCH();
        }

        // ---- correction entries ----
        S->n_corr = 0;
        if (nfail && S->contract && m <= (1u << 24) && nfail * n <= (1u << 24)) {
            // supports count every element: only the number of entries is reported
            WsBuf<uint32_t> seen(ws, m);
            BM_CUDA(cudaMemsetAsync(seen.p, 0, seen.bytes(), st));
            k_count_corrections<<<grid_for(32 * nfail), 256, 0, st>>>(S->d_fail_tid.p, nfail, S->d_bits.p, n, seen.p,
                                                                      &d_stat.p->ncorr);
            BM_CHECK_LAUNCH();
        } else if (nfail) {
            const uint64_t nwords = (m + 31) / 32;
            WsBuf<uint32_t> bits(ws, nwords);
            WsBuf<uint64_t> wrank(ws, nwords + 1), d_nu(ws, 1);
            BM_CUDA(cudaMemsetAsync(bits.p, 0, bits.bytes(), st));
            k_mark_failed<<<grid_for(nfail), 256, 0, st>>>(S->d_fail_tid.p, nfail, bits.p);
            BM_CHECK_LAUNCH();
            k_popc_words<<<grid_for(nwords), 256, 0, st>>>(bits.p, nwords, wrank.p);
            BM_CHECK_LAUNCH();
            scan_exclusive(wrank.p, nwords, d_nu.p, st);
            uint64_t nu = 0;
            BM_CUDA(cudaMemcpyAsync(&nu, d_nu.p, 8, cudaMemcpyDeviceToHost, st));
            BM_CUDA(cudaStreamSynchronize(st));
            WsBuf<uint64_t> fptr(ws, nu + 1), cursor(ws, nu + 1), d_sum(ws, 1);
            WsBuf<uint32_t> fitems(ws, nfail);
            BM_CUDA(cudaMemsetAsync(fptr.p, 0, fptr.bytes(), st));
            BM_CUDA(cudaMemsetAsync(cursor.p, 0, cursor.bytes(), st));
            k_count_per_tid<<<grid_for(nfail), 256, 0, st>>>(S->d_fail_tid.p, nfail, bits.p, wrank.p, fptr.p);
            BM_CHECK_LAUNCH();
            k_scan_single_block<<<1, SCAN_TPB, 0, st>>>(fptr.p, nu, d_sum.p, 1);
            BM_CHECK_LAUNCH();
            k_fill_per_tid<<<grid_for(nfail), 256, 0, st>>>(f_item.p, S->d_fail_tid.p, nfail, bits.p,
                                                           wrank.p, fptr.p,
                                                           (unsigned long long *)cursor.p, fitems.p);
            BM_CHECK_LAUNCH();
            k_corrections<false><<<nch, TPB, 0, st>>>(v, m, bits.p, wrank.p, fptr.p, fitems.p, &d_stat.p->ncorr,
                                                       nullptr);
            BM_CHECK_LAUNCH();
            if (!S->contract) {
                BM_CUDA(cudaMemcpyAsync(stat, d_stat.p, sizeof(BuildStat), cudaMemcpyDeviceToHost, st));
                BM_CUDA(cudaStreamSynchronize(st));
                if (stat->ncorr) {
                    S->d_corr.alloc(2 * stat->ncorr);
                    BM_CUDA(cudaMemsetAsync(&d_stat.p->ncorr, 0, 8, st));
                    k_corrections<true><<<nch, TPB, 0, st>>>(v, m, bits.p, wrank.p, fptr.p, fitems.p,
                                                              &d_stat.p->ncorr, S->d_corr.p);
                    BM_CHECK_LAUNCH();
                }
            }
        }
        if (nfail) {
            E.record(4, st);
            E.record(1, st);
            BM_CUDA(cudaMemcpyAsync(stat, d_stat.p, sizeof(BuildStat), cudaMemcpyDeviceToHost, st));
            BM_CUDA(cudaStreamSynchronize(st));
            S->n_corr = stat->ncorr;
        }
    }
    ws.done();
    S->timing.build_ms = E.ms(0, 1);
    S->timing.place_ms = E.ms(2, 3);
    S->timing.finalize_ms = E.ms(3, 4);
}

}  // namespace bm

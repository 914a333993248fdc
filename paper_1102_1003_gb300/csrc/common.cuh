// Shared helpers of the CUDA path: error plumbing, device utilities, layout
// arithmetic (Sec. III-A) and the internal representation of a built set.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "batmap.h"
#include "perm.cuh"

namespace bm {

// ---- error plumbing ---------------------------------------------------------

void set_error(const std::string &msg);

struct Error {
    batmap_status code;
    std::string msg;
};

#define BM_CUDA(call)                                                                       \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess) {                                                            \
            throw ::bm::Error{e_ == cudaErrorMemoryAllocation ? BATMAP_ERR_NOMEM            \
                                                              : BATMAP_ERR_CUDA,            \
                              std::string(#call) + ": " + cudaGetErrorString(e_)};         \
        }                                                                                   \
    } while (0)

void count_launch();
#define BM_CHECK_LAUNCH()             \
    do {                              \
        BM_CUDA(cudaGetLastError());  \
        ::bm::count_launch();         \
    } while (0)

#define BM_REQUIRE(cond, code, msg)                                                         \
    do {                                                                                    \
        if (!(cond)) throw ::bm::Error{(code), (msg)};                                      \
    } while (0)

// Device memory of the library.  Where there is none left, what it keeps for later
// calls (arrays of freed sets, idle call scratch) is given back and the request tried
// once more; then BATMAP_ERR_NOMEM.  batmap_test_memory_limit makes less of it.
void *device_alloc(size_t bytes);
void device_free(void *p, size_t bytes);
// Free memory and what the library keeps idle, so that a call finds the same before
// and after others that were freed.  Within a build only (the placement scratch is the build's).
uint64_t device_available();

// RAII device buffer.
template <typename T>
struct DevBuf {
    T *p = nullptr;
    size_t n = 0;
    DevBuf() = default;
    explicit DevBuf(size_t count) { alloc(count); }
    DevBuf(const DevBuf &) = delete;
    DevBuf &operator=(const DevBuf &) = delete;
    DevBuf(DevBuf &&o) noexcept : p(o.p), n(o.n) { o.p = nullptr; o.n = 0; }
    DevBuf &operator=(DevBuf &&o) noexcept {
        if (this != &o) { release(); p = o.p; n = o.n; o.p = nullptr; o.n = 0; }
        return *this;
    }
    ~DevBuf() { release(); }
    void alloc(size_t count) {
        release();
        if (count) p = static_cast<T *>(device_alloc(count * sizeof(T)));
        n = count;
    }
    void ensure(size_t count) { if (count > n) alloc(count); }
    void release() {
        if (p) device_free(p, n * sizeof(T));
        p = nullptr;
        n = 0;
    }
    size_t bytes() const { return n * sizeof(T); }
};

// The arrays of built sets come from a cache: a freed set's arrays (after a
// device synchronisation, as cudaFree would do) are kept for the next build, at
// most four of more than 64 MiB and 32 smaller ones, and a quarter of the device's
// memory in all, reused when no larger than twice the request plus 1 MiB.  A small build makes about thirty allocations,
// which cost more than its kernels.
uint8_t *bm_buffer_take(size_t bytes, size_t *capacity);
void bm_buffer_give(uint8_t *p, size_t capacity);
void bm_buffer_release_all();

// While one lives, arrays given back on this thread wait for no further work:
// its constructor has waited for all of the device's.
struct ReleaseScope {
    ReleaseScope();
    ~ReleaseScope();
};

template <typename T>
struct CacheBuf {
    T *p = nullptr;
    size_t n = 0, cap = 0;
    CacheBuf() = default;
    CacheBuf(const CacheBuf &) = delete;
    CacheBuf &operator=(const CacheBuf &) = delete;
    ~CacheBuf() { release(); }
    void alloc(size_t count) {
        release();
        if (count) p = reinterpret_cast<T *>(bm_buffer_take(count * sizeof(T), &cap));
        n = count;
    }
    void ensure(size_t count) { if (count > n) alloc(count); }
    void release() {
        if (p) bm_buffer_give(reinterpret_cast<uint8_t *>(p), cap);
        p = nullptr;
        n = cap = 0;
    }
};
using BmBuf = CacheBuf<uint8_t>;

// Device scratch of one call that synchronises its stream before it returns:
// pieces of an arena that the call holds alone and gives back (after waiting for
// the stream, unless done() says it has) to at most four kept for later calls,
// each of at most 256 MiB; batmap_release_scratch frees them.
struct Arena;
class Workspace {
  public:
    explicit Workspace(cudaStream_t st);
    ~Workspace();
    Workspace(const Workspace &) = delete;
    Workspace &operator=(const Workspace &) = delete;
    void *bytes(size_t count);  // nullptr for 0
    void *host();               // PINNED bytes of pinned host memory, for what the call reads back
    static constexpr size_t PINNED = 128 << 10;
    void done() { synced_ = true; }

  private:
    Arena *arena_;
    cudaStream_t st_;
    bool synced_ = false;
};
template <typename T>
struct WsBuf {
    T *p;
    size_t n;
    WsBuf(Workspace &w, size_t count) : p(static_cast<T *>(w.bytes(count * sizeof(T)))), n(count) {}
    size_t bytes() const { return n * sizeof(T); }
};
void release_arenas();

// Events bracketing phases of a call on its stream (kept for later sets).
struct PhaseEvents {
    static constexpr int N = 8;
    cudaEvent_t ev[N] = {};
    bool ok = false;
    void create();
    void record(int i, cudaStream_t st) { BM_CUDA(cudaEventRecord(ev[i], st)); }
    float ms(int a, int b) const {
        float t = 0.f;
        if (ok && cudaEventElapsedTime(&t, ev[a], ev[b]) != cudaSuccess) {
            cudaGetLastError();
            t = 0.f;
        }
        return t;
    }
    PhaseEvents() = default;
    PhaseEvents(const PhaseEvents &) = delete;
    PhaseEvents &operator=(const PhaseEvents &) = delete;
    ~PhaseEvents();
};

// ---- layout arithmetic (Sec. III-A) ----------------------------------------

// Slot of pi = pi_t(x) in table t of a BatMap with range r (power of two,
// >= r0 = 2^shift): |B_0| floor((pi mod r)/r0) + (pi mod r0) + t r0.
__host__ __device__ __forceinline__ uint64_t slot_of(uint32_t t, uint32_t pi, uint32_t r,
                                                    uint32_t shift) {
    uint32_t r0 = 1u << shift;
    uint32_t h = pi & (r - 1u);
    return 3ull * r0 * (uint64_t)(h >> shift) + (h & (r0 - 1u)) + (uint64_t)t * r0;
}

// ---- compare work units ----------------------------------------------------

// One unit of the all-pairs compare: rows [r0, r1) x columns [c0, c1) of the
// width-sorted item order, word range [k0, k0 + klen) of the column width.
// Rows are never wider than columns; columns of a unit share one width.
struct WorkUnit {
    uint32_t r0, r1, c0, c1;
    uint32_t k0, klen;
    uint32_t inst;   // instance index (batched launches), 0 otherwise
    uint32_t shape;  // tile shape index (0-based) | UNIT_WHOLE_K if [k0, k0+klen) is the whole width
};
constexpr uint32_t UNIT_WHOLE_K = 0x100u;  // the unit owns its pairs: plain stores, no atomics
constexpr uint32_t UNIT_SHAPE_MASK = 0xFFu;
static_assert(sizeof(WorkUnit) == 32, "WorkUnit layout");

// Per-instance device view used by the compare kernel (batched form indexes
// an array of these by WorkUnit::inst).
struct InstView {
    const uint4 *bm;          // BatMap bytes of this instance, as 16-byte chunks
    const uint32_t *line_off; // [n] sorted order: byte offset / 128 of each BatMap
    const uint32_t *wshift;   // [n] sorted order: e with |B|/4 words = 3 * 2^e
    const uint32_t *order;    // [n] sorted position -> original item id
    uint32_t *C;              // supports: packed upper triangle (original ids), or n_a x (n - n_a) in cross mode
    uint32_t n;
    uint32_t n_a;             // 0: all pairs i < j; else cross pairs of items [0, n_a) with [n_a, n)
    uint32_t shift;           // s: r_0 = 2^s, codes (pi >> s) + 1 (the probe route decodes slots)
};

// Index of the support of the pair of original items (oi, oj) in C.
__device__ __forceinline__ uint64_t support_index(uint32_t oi, uint32_t oj, uint64_t n, uint32_t n_a) {
    const uint64_t lo = oi < oj ? oi : oj, hi = oi < oj ? oj : oi;
    if (n_a) return lo * (n - n_a) + (hi - n_a);
    return lo * n - lo * (lo + 1) / 2 + (hi - lo - 1);
}

}  // namespace bm

// The library-owned handle behind the opaque C type.
struct batmap_set {
    batmap_params params{};
    uint32_t m = 0, n = 0, shift = 0, r0 = 0;

    // number of supports (pairs) the set reports
    uint64_t npairs() const { return n_a ? (uint64_t)n_a * (n - n_a) : (uint64_t)n * (n > 0 ? n - 1 : 0) / 2; }
    uint64_t n_elements = 0, bytes = 0, n_failed = 0, n_corr = 0;
    double word_pairs = 0.0;
    double probe_word_pairs = 0.0;  // part of word_pairs counted by the probe route (scan-equivalent words)
    double probe_words = 0.0;       // words the probe route reads: rows' widths x columns per unit
    uint32_t n_a = 0;            // cross mode: items [0, n_a) x [n_a, n); 0 = all pairs
    uint32_t d = 2;              // copies per element: 2 (2-of-3 BatMaps) or 3 (3-of-4, k-way witnesses)
    uint64_t gen = 0;            // unique build id (batch plans key on it)
    bool skip_schedule = false;  // pool builds need no all-pairs schedule
    cudaStream_t stream = nullptr;

    // host metadata
    std::vector<uint32_t> range;          // r_i, original order
    std::vector<uint32_t> order;          // sorted position -> original id
    std::vector<uint32_t> rank;           // original id -> sorted position
    std::vector<uint64_t> byte_off;       // byte offset of BatMap, sorted order
    std::vector<uint32_t> wshift_sorted;  // e per sorted position
    std::vector<uint32_t> class_begin;    // sorted positions where a width class starts (+ n)
    std::vector<bm::WorkUnit> units;      // compare schedule, longest first (contract: made when asked for)

    // device data
    bm::BmBuf d_bm;                       // all BatMaps, width-sorted order
    bool contract = false;                // pair supports by the contraction of bit rows (dense.cu)
    bool mm_add = false;                  // its units add into zeroed supports
    uint32_t mm_count = 0, kblocks = 0;
    bm::BmBuf d_bits;                     // bit rows, original item order
    bm::BmBuf d_mm;                       // queue counter, timeout flag, number of pairs (64 bytes); the units
    bm::CacheBuf<uint32_t> d_meta;          // the per-item arrays of the build, one upload
    struct DevPtr { uint32_t *p = nullptr; };
    DevPtr d_line_off;                    // [n] sorted (in d_meta, as the next two)
    DevPtr d_wshift;                      // [n] sorted
    DevPtr d_order;                       // [n]
    bm::CacheBuf<bm::WorkUnit> d_units;
    bm::CacheBuf<uint32_t> d_corr;          // [2 * n_corr] (i, j) original ids, i < j
    bm::CacheBuf<uint64_t> d_fail_off;      // [n+1] failed tids per item (CSR)
    bm::CacheBuf<uint32_t> d_fail_tid;      // [n_failed], sorted per item
    // 3-of-4 sets (original item order): byte offsets, log2 r_i, own copy of pi_0..pi_3
    bm::CacheBuf<uint64_t> d_base;          // [n+1]
    bm::CacheBuf<uint32_t> d_rlog;          // [n]
    bm::CacheBuf<uint32_t> d_perm;          // [4 m] copy of the caller's table, if one was given
    bm::PermView perm{};                  // the set's pi_t (table view or computed)

    // timing of the most recent calls
    bm::PhaseEvents build_ev, pairs_ev;
    batmap_timing timing{};

    // scratch reused across pair_support_all calls
    bm::CacheBuf<uint32_t> d_C;             // packed upper triangle when no d_full
    bm::CacheBuf<uint32_t> d_counters;      // work-queue counter
    bm::CacheBuf<bm::InstView> d_view;      // device copy of this set's InstView
    bm::CacheBuf<uint64_t> d_blocksums;     // compaction tile states
    bm::CacheBuf<uint64_t> d_total;         // compaction total
};

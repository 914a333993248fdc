// Bit rows of a set family (Sec. I-B, the bitmap vertical representation) and
// the contraction of such rows on the tensor cores.
#pragma once

#include "common.cuh"

namespace bm {

// One bit per (item, transaction); bit x of item i sits in block kb = x / 256
// at word (x / 32) mod 8 of the 32 bytes at i * row_stride + kb * kb_stride.
// Pair sets keep block after block (rows of a block contiguous: a tile's rows
// are one bulk copy, row_stride 32); sets for k-way supports keep row after
// row (kb_stride 32).
constexpr uint32_t BITS_K = 256;
inline uint32_t bits_blocks(uint32_t m) { return (m + BITS_K - 1) / BITS_K; }

struct BitsLayout {
    uint64_t row_stride, kb_stride;
    uint32_t kblocks;
};
inline BitsLayout bits_block_major(uint32_t n, uint32_t m) { return {32, 32ull * n, bits_blocks(m)}; }
inline BitsLayout bits_row_major(uint32_t m) { return {32ull * bits_blocks(m), 32, bits_blocks(m)}; }

// Writes every block of the n rows (no zeroing needed before).  d_flags[0] <-
// 1 if a tid >= m was seen (and skipped), d_flags[1] <- 1 if some tidlist is
// not strictly increasing; the caller zeroes both.  The rows are right either
// way, unless `sorted_only` leaves out the pass that serves unsorted lists
// (for callers that refuse them).
void enqueue_bits(const uint64_t *d_off, const uint32_t *d_tids, uint32_t n, uint32_t m, const BitsLayout &L,
                  uint8_t *d_bits, int *d_flags, bool sorted_only, cudaStream_t st);

// Allocates `bytes` of bit rows unless they would take more than half of the
// memory that no caller and no set holds, less the `supports` bytes that the set's
// calls may ask for; false (and no rows) if so, or if the allocation fails.
// Called within a build.
bool take_bits(BmBuf *buf, uint64_t bytes, uint64_t supports);

// |S_a1 cap .. cap S_ak| of nq queries of k ids each (1 <= k <= 4) over
// row-major bit rows: AND and popcount.
void enqueue_bits_support(const uint8_t *d_bits, uint32_t kblocks, uint32_t k, const uint32_t *d_items, uint64_t nq,
                          uint32_t *d_support, cudaStream_t st);

// ---- contraction -----------------------------------------------------------------

struct MmView {          // one instance
    const uint8_t *bits; // block-major rows
    uint32_t *C;         // supports: packed upper triangle, or n_a x (n - n_a)
    uint32_t n, n_a;
};
struct MmUnit {          // 256 rows x MM_COLS columns over the K blocks [kb0, kb1)
    uint32_t r0, c0, kb0, kb1;
    uint32_t inst;
    uint32_t add;        // 1: partial sums, added into zeroed supports; 0: stored
    uint32_t pad[2];
};
static_assert(sizeof(MmUnit) == 32, "MmUnit layout");
constexpr uint32_t MM_ROWS = 256, MM_COLS = 240;

// Estimated seconds of the contraction of n rows (cross: n_a x (n - n_a)).
double contract_seconds(uint32_t n, uint32_t n_a, uint32_t kblocks);
// Appends the units of one instance; true if they add (C must be zeroed).
// others: seconds of work of the other instances of the launch.
bool contract_units(uint32_t n, uint32_t n_a, uint32_t kblocks, uint32_t inst, double others,
                    std::vector<MmUnit> *out);
void prepare_contract();  // kernel attributes (before stream capture)
// One persistent launch over the units (longest first), of the instances at
// d_views or, if that is NULL, of `one`.  d_state: two zeroed words, [0] the
// queue counter, [1] <- 1 if a bounded wait gave up.
void launch_contract(const MmView *d_views, const MmView &one, const MmUnit *d_units, uint32_t count,
                     uint32_t *d_state, cudaStream_t st, unsigned long long *d_stamps = nullptr,
                     uint32_t test_spin = 0);

// Decides whether a set's pair supports come from its bit rows; if so, allocates
// them and enqueues their build (d_flags as in enqueue_bits) and the units.
void plan_contract(batmap_set *S, const uint64_t *d_off, const uint32_t *d_tids, int *d_flags, bool sorted_only,
                   cudaStream_t st);
// Supports of all pairs of a set planned that way into C.
void enqueue_contract(batmap_set *S, uint32_t *C, cudaStream_t st);
MmView contract_view(const batmap_set *S, uint32_t *C);

}  // namespace bm

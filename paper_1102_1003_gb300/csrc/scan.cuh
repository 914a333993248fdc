// Block- and device-level prefix sums used for ordered stream compaction
// (failed-insertion lists, frequent-pair output) and bitmap ranks.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace bm {

constexpr int SCAN_TPB = 256;

// Exclusive prefix of `v` over the threads of a 256-thread block, in thread
// order.  Returns the prefix; *total receives the block sum.  All threads of
// the block must call it (contains __syncthreads).
__device__ __forceinline__ uint64_t block_exclusive_scan(uint64_t v, uint64_t *total) {
    __shared__ uint64_t warp_sums[SCAN_TPB / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        uint64_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint64_t w = lane < SCAN_TPB / 32 ? warp_sums[lane] : 0;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            uint64_t y = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += y;
        }
        if (lane < SCAN_TPB / 32) warp_sums[lane] = w;
    }
    __syncthreads();
    uint64_t warp_prefix = warp ? warp_sums[warp - 1] : 0;
    *total = warp_sums[SCAN_TPB / 32 - 1];
    __syncthreads();
    return warp_prefix + x - v;
}

// ---- decoupled look-back over tiles (Merrill and Garland) ----
// A tile's state word: 0 (not known), STATE_SUM | its sum, or STATE_PREFIX | the
// sum up to and with it.
constexpr uint64_t STATE_SUM = 1ull << 62, STATE_PREFIX = 2ull << 62, STATE_VALUE = STATE_SUM - 1;
constexpr uint32_t LOOKBACK_SPINS = 1u << 24;

// Sum of the tiles before `tile` by the first warp (all lanes): looks back 32
// states at a time.  ~0 if a predecessor's state did not come (bounded; the
// predecessors run, as tiles are handed out in order).
__device__ __forceinline__ uint64_t look_back(uint64_t *state, uint64_t tile, uint32_t lane) {
    uint64_t sum = 0;
    for (int64_t last = (int64_t)tile - 1; last >= 0; last -= 32) {
        const int64_t at = last - lane;
        uint64_t v = at < 0 ? STATE_PREFIX : 0;
        for (uint32_t it = 0; !(v >> 62); it++) {
            if (it == LOOKBACK_SPINS) break;
            v = *(volatile uint64_t *)&state[at];
        }
        if (!__all_sync(0xffffffffu, (v >> 62) != 0)) return ~0ull;
        const uint32_t done = __ballot_sync(0xffffffffu, (v >> 62) == 2);
        const uint32_t upto = done ? __ffs(done) - 1 : 31;  // lanes behind a prefix do not count
        uint64_t x = lane <= upto ? v & STATE_VALUE : 0;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
        sum += x;
        if (done) break;
    }
    return sum;
}

// In-place exclusive scan of a[0..count) by ONE block of 256 threads; writes
// the grand total to *total (device) and a[count] if with_tail.
__global__ void k_scan_single_block(uint64_t *a, uint64_t count, uint64_t *total, int with_tail);

// Exclusive scan of a uint64 array on `stream`: a[i] <- sum_{j<i} a[j], a[count]
// and *d_total (if not NULL) <- the sum (~0: a bounded wait gave up; check_total).
// One block up to SCAN_ONE values (1.5 us per 2,048), above
// it tiles with look-back (136,492 values: 50 us by one block).  `state`: room for
// scan_states(count) words.
constexpr uint64_t SCAN_ONE = 8192;
inline uint64_t scan_states(uint64_t count) { return count > SCAN_ONE ? (count + 2047) / 2048 + 1 : 0; }
void scan_with_tail(uint64_t *d_a, uint64_t count, uint64_t *d_total, uint64_t *state, cudaStream_t stream);

// a[i] <- sum_{j<i} a[j]; *d_total <- sum.  Uses one block.
void scan_exclusive(uint64_t *d_a, uint64_t count, uint64_t *d_total, cudaStream_t stream);

void check_total(uint64_t total);  // throws BATMAP_ERR_TIMEOUT for ~0

}  // namespace bm

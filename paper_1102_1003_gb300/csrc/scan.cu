#include "common.cuh"
#include "scan.cuh"

namespace bm {

__global__ void k_scan_single_block(uint64_t *a, uint64_t count, uint64_t *total, int with_tail) {
    constexpr int PER = 8;  // values per thread per tile
    uint64_t carry = 0;
    for (uint64_t base = 0; base < count; base += (uint64_t)SCAN_TPB * PER) {
        uint64_t v[PER];
        uint64_t sum = 0;
        uint64_t i0 = base + (uint64_t)threadIdx.x * PER;
#pragma unroll
        for (int q = 0; q < PER; q++) {
            v[q] = (i0 + q < count) ? a[i0 + q] : 0;
            sum += v[q];
        }
        uint64_t tile_total;
        uint64_t pre = block_exclusive_scan(sum, &tile_total) + carry;
#pragma unroll
        for (int q = 0; q < PER; q++) {
            if (i0 + q < count) a[i0 + q] = pre;
            pre += v[q];
        }
        carry += tile_total;
    }
    if (threadIdx.x == 0) {
        if (total) *total = carry;
        if (with_tail) a[count] = carry;
    }
}

// state: one zeroed word per tile of 2,048 values, then the zeroed tile counter.
__global__ void __launch_bounds__(SCAN_TPB) k_scan_tiles(uint64_t *a, uint64_t count, uint64_t *total, uint64_t *state,
                                                         uint64_t tiles) {
    constexpr int PER = 8;
    __shared__ uint64_t s_tile, s_before;
    const uint32_t lane = threadIdx.x & 31u;
    if (threadIdx.x == 0) s_tile = atomicAdd((unsigned long long *)&state[tiles], 1ull);
    __syncthreads();
    const uint64_t tile = s_tile, i0 = tile * (SCAN_TPB * PER) + (uint64_t)threadIdx.x * PER;
    uint64_t v[PER], sum = 0;
#pragma unroll
    for (int q = 0; q < PER; q++) {
        v[q] = i0 + q < count ? a[i0 + q] : 0;
        sum += v[q];
    }
    uint64_t all;
    const uint64_t mine = block_exclusive_scan(sum, &all);
    if (threadIdx.x < 32) {
        if (lane == 0 && tile) *(volatile uint64_t *)&state[tile] = STATE_SUM | all;
        const uint64_t before = look_back(state, tile, lane);
        if (lane == 0) {
            if (before != ~0ull) *(volatile uint64_t *)&state[tile] = STATE_PREFIX | (before + all);
            s_before = before;
            if (tile + 1 == tiles || before == ~0ull) {
                const uint64_t t = before == ~0ull ? ~0ull : before + all;
                if (total) *(volatile uint64_t *)total = t;
                if (tile + 1 == tiles) a[count] = t;
            }
        }
    }
    __syncthreads();
    if (s_before == ~0ull) return;
    uint64_t pre = s_before + mine;
#pragma unroll
    for (int q = 0; q < PER; q++) {
        if (i0 + q < count) a[i0 + q] = pre;
        pre += v[q];
    }
}

void scan_with_tail(uint64_t *d_a, uint64_t count, uint64_t *d_total, uint64_t *state, cudaStream_t stream) {
    if (count <= SCAN_ONE) {
        k_scan_single_block<<<1, SCAN_TPB, 0, stream>>>(d_a, count, d_total, 1);
    } else {
        const uint64_t tiles = scan_states(count) - 1;
        BM_CUDA(cudaMemsetAsync(state, 0, (tiles + 1) * sizeof(uint64_t), stream));
        k_scan_tiles<<<(unsigned)tiles, SCAN_TPB, 0, stream>>>(d_a, count, d_total, state, tiles);
    }
    BM_CHECK_LAUNCH();
}

void scan_exclusive(uint64_t *d_a, uint64_t count, uint64_t *d_total, cudaStream_t stream) {
    k_scan_single_block<<<1, SCAN_TPB, 0, stream>>>(d_a, count, d_total, 0);
    BM_CHECK_LAUNCH();
}

}  // namespace bm

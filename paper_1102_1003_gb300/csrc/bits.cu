// Bit rows from CSR tidlists (the bitmap vertical representation, Sec. I-B).
//
// One warp writes one item's bits of one 32,768-transaction chunk: it finds
// the chunk's tids by two 32-way searches (about log32 |S| dependent reads),
// ORs them into 4 KiB of shared memory and stores the 128 blocks of 32 bytes.
// Every byte of the matrix is written once, so nothing is zeroed before, no
// global atomic is used and the lists' order is checked on the way.
// Bound: HBM, 4 bytes read per tid and 1 bit written per (item, transaction).
#include <algorithm>

#include "bits.cuh"

namespace bm {

constexpr uint32_t CHUNK_KB = 128;                   // blocks per warp
constexpr uint32_t CHUNK_BITS = CHUNK_KB * BITS_K;   // 32,768
constexpr int BW = 8;                                // warps per CTA

// First index in a[0 .. n) whose value is >= v, by the whole warp.  A function
// of the list and v alone, so neighbouring chunks agree on their border even
// when the list is not sorted.
__device__ __forceinline__ uint64_t warp_lower_bound(const uint32_t *__restrict__ a, uint64_t n, uint32_t v,
                                                     uint32_t lane) {
    uint64_t lo = 0, hi = n;
    while (lo < hi) {
        const uint64_t step = (hi - lo + 31) >> 5;
        const uint64_t p = lo + lane * step + (step - 1);
        const bool below = p < hi && __ldg(&a[p]) < v;
        const uint32_t c = __popc(__ballot_sync(0xffffffffu, below));
        const uint64_t top = lo + c * step + (step - 1);  // the first probe not below, if c < 32
        lo = min(lo + c * step, hi);
        if (c < 32) hi = min(hi, top);
    }
    return lo;
}

__global__ void __launch_bounds__(32 * BW)
k_bits(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tids, uint32_t n, uint32_t m, BitsLayout L,
       uint8_t *__restrict__ out, int *__restrict__ flags) {
    __shared__ __align__(16) uint32_t s_bits[BW][CHUNK_BITS / 32];
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t *bits = s_bits[threadIdx.x >> 5];
    uint4 *bits4 = reinterpret_cast<uint4 *>(bits);
    const uint32_t nchunk = (L.kblocks + CHUNK_KB - 1) / CHUNK_KB;
    const uint64_t tasks = (uint64_t)n * nchunk, warps = (uint64_t)gridDim.x * BW;
    bool bad_tid = false, unsorted = false;
    // neighbouring warps: neighbouring items of the same chunk, whose 32-byte pieces share lines
    for (uint64_t w = blockIdx.x * (uint64_t)BW + (threadIdx.x >> 5); w < tasks; w += warps) {
        const uint32_t item = (uint32_t)(w % n), chunk = (uint32_t)(w / n);
#pragma unroll
        for (uint32_t j = 0; j < CHUNK_BITS / 32 / 4; j += 32) bits4[j + lane] = make_uint4(0, 0, 0, 0);
        const uint64_t b = off[item], size = off[item + 1] - b;
        const uint32_t *a = tids + b;
        const uint32_t x0 = chunk * CHUNK_BITS, x1 = x0 + CHUNK_BITS;  // m <= 2^30: no overflow
        const bool last = chunk + 1 == nchunk;
        const uint64_t e0 = chunk ? warp_lower_bound(a, size, x0, lane) : 0;
        const uint64_t e1 = last ? size : warp_lower_bound(a, size, x1, lane);
        unsorted |= e1 < e0;
        __syncwarp();
        for (uint64_t e = e0; e < e1; e += 128) {
            uint32_t x[4], y[4];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const uint64_t i = e + 32u * q + lane;
                x[q] = i < e1 ? __ldg(&a[i]) : 0xFFFFFFFFu;
                y[q] = i < e1 && i + 1 < size ? __ldg(&a[i + 1]) : 0xFFFFFFFFu;
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                if (e + 32u * q + lane >= e1) continue;
                unsorted |= !(x[q] < y[q]);
                if (x[q] >= m) bad_tid = true;
                else if (x[q] - x0 < CHUNK_BITS) atomicOr(&bits[(x[q] - x0) >> 5], 1u << (x[q] & 31u));
                else unsorted = true;
            }
        }
        __syncwarp();
        uint8_t *row = out + item * L.row_stride;
        const uint32_t kb0 = chunk * CHUNK_KB;
#pragma unroll
        for (uint32_t j = 0; j < CHUNK_KB * 2; j += 32) {
            const uint32_t i = j + lane, kb = kb0 + (i >> 1);
            if (kb < L.kblocks) *reinterpret_cast<uint4 *>(row + kb * L.kb_stride + 16u * (i & 1u)) = bits4[i];
        }
        __syncwarp();
    }
    if (bad_tid) atomicExch(&flags[0], 1);
    if (unsorted) atomicExch(&flags[1], 1);
}

// Adds the tids of lists that are not sorted (the chunk search finds those of
// sorted lists only).  Does nothing unless flags[1] is set.
__global__ void k_bits_unsorted(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tids, uint32_t n,
                                uint32_t m, BitsLayout L, uint8_t *__restrict__ out, int *__restrict__ flags) {
    if (!flags[1]) return;
    for (uint32_t i = blockIdx.y; i < n; i += gridDim.y) {
        const uint64_t b = off[i], e = off[i + 1];
        for (uint64_t k = b + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < e;
             k += (uint64_t)gridDim.x * blockDim.x) {
            const uint32_t x = tids[k];
            if (x >= m) {
                atomicExch(&flags[0], 1);
                continue;
            }
            uint32_t *w = reinterpret_cast<uint32_t *>(out + i * L.row_stride + (x >> 8) * L.kb_stride) + ((x >> 5) & 7u);
            atomicOr(w, 1u << (x & 31u));
        }
    }
}

void enqueue_bits(const uint64_t *d_off, const uint32_t *d_tids, uint32_t n, uint32_t m, const BitsLayout &L,
                  uint8_t *d_bits, int *d_flags, bool sorted_only, cudaStream_t st) {
    if (!n) return;
    const uint64_t tasks = (uint64_t)n * ((L.kblocks + CHUNK_KB - 1) / CHUNK_KB);
    const unsigned grid = (unsigned)std::min<uint64_t>((tasks + BW - 1) / BW, 1u << 20);
    k_bits<<<grid, 32 * BW, 0, st>>>(d_off, d_tids, n, m, L, d_bits, d_flags);
    BM_CHECK_LAUNCH();
    if (!sorted_only) {
        k_bits_unsorted<<<dim3(8, std::min<uint32_t>(n, 128u)), 256, 0, st>>>(d_off, d_tids, n, m, L, d_bits, d_flags);
        BM_CHECK_LAUNCH();
    }
}

}  // namespace bm

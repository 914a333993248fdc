// Failure correction and support-threshold compaction (Sec. III-C; Sec. I
// problem statement: report the pairs with support at least s).
//
// Supports live in a packed row-major upper triangle indexed by ORIGINAL item
// ids, so lexicographic (i, j) order is plain array order and the frequent
// pairs come out of one ordered stream compaction: every block takes the next
// tile of 4,096 supports, counts its qualifying ones, finds how many lie before
// the tile from its predecessors' states (decoupled look-back: Merrill and
// Garland, "Single-pass parallel prefix scan with decoupled look-back") and
// writes its triples through shared memory, 12 consecutive bytes each.
// Bound: HBM, 4 bytes read per pair and 12 written per frequent pair.  Before,
// a count pass, a scan and a write pass that ranked 256 supports at a time and
// searched each one's row: 598 us for 32 M pairs of n = 8,000, all frequent
// (512 MB: 76 us at the copy rate); this one 218 us with 72 registers, three blocks
// per SM that wait at their barriers, and about 175 with 48 and 32-bit row borders.
#include <algorithm>

#include "common.cuh"
#include "scan.cuh"

namespace bm {

constexpr int CTPB = SCAN_TPB;
constexpr int CQ = 4;                                // 16-byte loads per thread
constexpr uint32_t CCHUNK = CTPB * 4 * CQ;           // 4,096 supports per tile
constexpr uint32_t CSTAGE = CCHUNK / 2;              // triples staged at a time

__global__ void k_apply_corrections(const uint32_t *__restrict__ corr, uint64_t ncorr, uint64_t n,
                                    uint32_t n_a, uint32_t *__restrict__ C) {
    for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < ncorr;
         k += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t i = corr[2 * k], j = corr[2 * k + 1];
        if (n_a && !(i < n_a && j >= n_a)) continue;  // cross mode: A x B pairs only
        atomicAdd(&C[support_index(i, j, n, n_a)], 1u);
    }
}

// First packed index of row i: triangle i n - i (i + 1) / 2, rectangle i n_b.
__device__ __forceinline__ uint64_t row_start(uint64_t i, uint64_t n, uint32_t n_a) {
    return n_a ? i * (n - n_a) : i * n - i * (i + 1) / 2;
}

// Row of packed index L among [lo, hi].
__device__ __forceinline__ uint32_t row_of(uint64_t L, uint64_t n, uint32_t n_a, uint32_t lo, uint32_t hi) {
    while (lo < hi) {
        const uint32_t mid = lo + (hi - lo + 1) / 2;
        if (row_start(mid, n, n_a) <= L) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// state: one zeroed word per tile, then the zeroed tile counter.  *total <- the
// number of qualifying pairs (~0: a bounded wait gave up).  out may be NULL.
__global__ void __launch_bounds__(CTPB, 5) k_threshold(const uint32_t *__restrict__ C, uint64_t npairs, uint64_t n,
                                                    uint32_t n_a, uint32_t s, uint64_t *__restrict__ state,
                                                    uint64_t tiles, uint32_t *__restrict__ out, uint64_t cap,
                                                    uint64_t *__restrict__ total) {
    __shared__ uint32_t s_out[3 * CSTAGE];
    __shared__ uint64_t s_tile, s_before;
    __shared__ uint32_t s_rows[2];
    const uint32_t lane = threadIdx.x & 31u;
    if (threadIdx.x == 0) s_tile = atomicAdd((unsigned long long *)&state[tiles], 1ull);
    __syncthreads();
    const uint64_t tile = s_tile, base = tile * CCHUNK;
    if (threadIdx.x >= 32 && threadIdx.x < 34) {  // rows of the tile's first and last support
        const uint64_t L = threadIdx.x == 32 ? base : min(base + CCHUNK, npairs) - 1;
        s_rows[threadIdx.x - 32] = row_of(L, n, n_a, 0, n_a ? n_a - 1 : (uint32_t)n - 2);
    }
    // thread t holds the supports base + 1024 q + 4 t + j
    uint32_t v[CQ][4];
    uint64_t packed = 0;  // per q, the thread's number of qualifying supports (16 bits each)
    const bool vec = (reinterpret_cast<uintptr_t>(C) & 15u) == 0;
    uint32_t keep = 0;
#pragma unroll
    for (int q = 0; q < CQ; q++) {
        const uint64_t L = base + 1024u * q + 4u * threadIdx.x;
        if (vec && L + 4 <= npairs) {
            const uint4 x = __ldg(reinterpret_cast<const uint4 *>(C + L));
            v[q][0] = x.x; v[q][1] = x.y; v[q][2] = x.z; v[q][3] = x.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++) v[q][j] = L + j < npairs ? __ldg(&C[L + j]) : 0;
        }
#pragma unroll
        for (int j = 0; j < 4; j++) keep |= (v[q][j] >= s && L + j < npairs ? 1u : 0u) << (4 * q + j);
        packed |= (uint64_t)__popc((keep >> (4 * q)) & 15u) << (16 * q);
    }
    uint64_t sums;
    const uint64_t pre = block_exclusive_scan(packed, &sums);  // four 16-bit scans (<= 1024 each)
    const uint32_t count = (uint32_t)((sums & 0xFFFF) + ((sums >> 16) & 0xFFFF) + ((sums >> 32) & 0xFFFF) + (sums >> 48));
    if (threadIdx.x < 32) {
        if (lane == 0 && tile)
            *(volatile uint64_t *)&state[tile] = STATE_SUM | count;
        const uint64_t before = look_back(state, tile, lane);
        if (lane == 0) {
            if (before != ~0ull) *(volatile uint64_t *)&state[tile] = STATE_PREFIX | (before + count);
            s_before = before;
            if (tile + 1 == tiles || before == ~0ull) *(volatile uint64_t *)total = before == ~0ull ? ~0ull : before + count;
        }
    }
    __syncthreads();
    const uint64_t before = s_before;
    if (before == ~0ull || !out || before >= cap || !count) return;
    const uint32_t room = (uint32_t)min((uint64_t)count, cap - before);
    const uint32_t r0 = s_rows[0], r1 = s_rows[1];
    for (uint32_t p0 = 0; p0 < room; p0 += CSTAGE) {
        uint32_t first = 0;  // rank of the q-th kilobyte's first qualifying support
#pragma unroll
        for (int q = 0; q < CQ; q++) {
            uint32_t rank = first + (uint32_t)((pre >> (16 * q)) & 0xFFFF);
            const uint32_t bits = (keep >> (4 * q)) & 15u;
            if (bits && rank < p0 + CSTAGE && rank + 4 > p0) {
                const uint64_t L = base + 1024u * q + 4u * threadIdx.x;
                const uint32_t p = 1024u * q + 4u * threadIdx.x;  // its place in the tile
                uint32_t i = row_of(L, n, n_a, r0, r1);
                // starts of its row (modulo 2^32) and of the next, from the tile's first place on
                uint32_t here = (uint32_t)(row_start(i, n, n_a) - base);
                uint32_t next = i < r1 ? (uint32_t)(row_start(i + 1ull, n, n_a) - base) : CCHUNK;
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    while (p + j >= next && i < r1) {
                        i++;
                        here = next;
                        next = i < r1 ? (uint32_t)(row_start(i + 1ull, n, n_a) - base) : CCHUNK;
                    }
                    if ((bits >> j) & 1u) {
                        if (rank >= p0 && rank < p0 + CSTAGE) {
                            uint32_t *o = s_out + 3 * (rank - p0);
                            o[0] = i;
                            o[1] = p + j - here + (n_a ? 0 : i + 1);  // B items count from 0
                            o[2] = v[q][j];
                        }
                        rank++;
                    }
                }
            }
            first += (uint32_t)((sums >> (16 * q)) & 0xFFFF);
        }
        __syncthreads();
        const uint32_t words = 3 * min(room - p0, CSTAGE);
        uint32_t *o = out + 3 * (before + p0);
        for (uint32_t w = threadIdx.x; w < words; w += CTPB) o[w] = s_out[w];
        __syncthreads();
    }
}

// Tiles of the threshold compaction of npairs supports.
static uint64_t tiles_of(uint64_t npairs) { return (npairs + CCHUNK - 1) / CCHUNK; }

// Allocates the compaction scratch of a set ahead of stream capture.
void prepare_compaction(batmap_set *S) {
    if (S->npairs()) S->d_blocksums.ensure(tiles_of(S->npairs()) + 1);
}

static void enqueue_compaction(const uint32_t *C, uint64_t npairs, uint64_t n, uint32_t n_a, uint32_t s,
                               uint32_t *d_pairs, uint64_t cap, uint64_t *state, uint64_t *d_total, cudaStream_t st) {
    if (npairs == 0) {
        BM_CUDA(cudaMemsetAsync(d_total, 0, sizeof(uint64_t), st));
        return;
    }
    const uint64_t tiles = tiles_of(npairs);
    BM_CUDA(cudaMemsetAsync(state, 0, (tiles + 1) * sizeof(uint64_t), st));
    k_threshold<<<(unsigned)tiles, CTPB, 0, st>>>(C, npairs, n, n_a, s, state, tiles, cap ? d_pairs : nullptr, cap,
                                                  d_total);
    BM_CHECK_LAUNCH();
}

// Enqueues the correction and the compaction of one set: adds the correction
// entries into C, writes the frequent pairs (at most cap) and stores their
// number at d_total (~0: see check_total).  No host synchronisation.
void enqueue_correct_compact(batmap_set *S, uint32_t *C, uint32_t s, uint32_t *d_pairs, uint64_t cap,
                             uint64_t *d_total, cudaStream_t st) {
    if (S->n_corr && !S->contract) {  // the contraction counts every element
        uint64_t g = std::min<uint64_t>((S->n_corr + 255) / 256, 1u << 16);
        k_apply_corrections<<<(unsigned)g, 256, 0, st>>>(S->d_corr.p, S->n_corr, S->n, S->n_a, C);
        BM_CHECK_LAUNCH();
    }
    prepare_compaction(S);
    enqueue_compaction(C, S->npairs(), S->n, S->n_a, s, d_pairs, cap, S->d_blocksums.p, d_total, st);
}

// Number of tile states the threshold compaction of n items needs (and one
// more word, the tile counter).
uint64_t threshold_blocks(uint64_t n) { return tiles_of(n * (n > 0 ? n - 1 : 0) / 2); }

// Threshold compaction of a packed support triangle that no set owns, with
// threshold_blocks(n) + 1 words of state provided by the caller; allocates nothing.
void enqueue_threshold_into(const uint32_t *C, uint64_t n, uint32_t s, uint32_t *d_pairs, uint64_t cap,
                            uint64_t *state, uint64_t *d_total, cudaStream_t st) {
    enqueue_compaction(C, n * (n > 0 ? n - 1 : 0) / 2, n, 0, s, d_pairs, cap, state, d_total, st);
}

// The same for the dense path, the state in a buffer the library grows.
void enqueue_threshold(const uint32_t *C, uint64_t n, uint32_t s, uint32_t *d_pairs, uint64_t cap,
                       DevBuf<uint64_t> *state, uint64_t *d_total, cudaStream_t st) {
    state->ensure(threshold_blocks(n) + 1);
    enqueue_threshold_into(C, n, s, d_pairs, cap, state->p, d_total, st);
}

void check_total(uint64_t total) {
    BM_REQUIRE(total != ~0ull, BATMAP_ERR_TIMEOUT, "compaction: a bounded wait between thread blocks timed out");
}

}  // namespace bm

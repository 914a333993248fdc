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
// per SM that wait at their barriers, 177 with 48 and 32-bit row borders, 167 with a
// stage of each warp's own, behind no barrier but those of the count.
#include <algorithm>

#include "common.cuh"
#include "scan.cuh"

namespace bm {

constexpr int CTPB = SCAN_TPB;
constexpr int CQ = 4;                                // 16-byte loads per thread
constexpr uint32_t CCHUNK = CTPB * 4 * CQ;           // 4,096 supports per tile
constexpr uint32_t CWARPS = CTPB / 32;
constexpr uint32_t CSTAGE = 128;                     // triples that a warp stages at a time

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
    __shared__ uint32_t s_out[CWARPS][3 * CSTAGE];
    __shared__ uint64_t s_tile, s_before;
    __shared__ uint32_t s_rows[2], s_count[CWARPS];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_tile = atomicAdd((unsigned long long *)&state[tiles], 1ull);
    __syncthreads();
    const uint64_t tile = s_tile, base = tile * CCHUNK;
    if (threadIdx.x >= 32 && threadIdx.x < 34) {  // rows of the tile's first and last support
        const uint64_t L = threadIdx.x == 32 ? base : min(base + CCHUNK, npairs) - 1;
        s_rows[threadIdx.x - 32] = row_of(L, n, n_a, 0, n_a ? n_a - 1 : (uint32_t)n - 2);
    }
    // a lane holds the supports base + place + 128 q + j
    const uint32_t place = CSTAGE * CQ * warp + 4u * lane;
    uint32_t v[CQ][4];
    uint64_t packed = 0;  // per q, the lane's number of qualifying supports (16 bits each)
    const bool vec = (reinterpret_cast<uintptr_t>(C) & 15u) == 0;
    uint32_t keep = 0;
#pragma unroll
    for (int q = 0; q < CQ; q++) {
        const uint64_t L = base + place + CSTAGE * q;
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
    uint64_t pre = packed;  // four 16-bit scans over the warp (<= 128 each)
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, pre, d);
        if (lane >= (uint32_t)d) pre += y;
    }
    const uint64_t sums = __shfl_sync(0xffffffffu, pre, 31);
    pre -= packed;
    if (lane == 0)
        s_count[warp] = (uint32_t)((sums & 0xFFFF) + ((sums >> 16) & 0xFFFF) + ((sums >> 32) & 0xFFFF) + (sums >> 48));
    __syncthreads();
    uint32_t count = 0, ahead = 0;  // the tile's, and those of the warps before
#pragma unroll
    for (uint32_t w = 0; w < CWARPS; w++) {
        ahead += w < warp ? s_count[w] : 0;
        count += s_count[w];
    }
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
    const uint32_t r0 = s_rows[0], r1 = s_rows[1];
    uint64_t to = before + ahead;  // the warp's next triple
    uint32_t *stage = s_out[warp];
#pragma unroll
    for (int q = 0; q < CQ; q++) {
        const uint32_t found = (uint32_t)(sums >> (16 * q)) & 0xFFFF, bits = (keep >> (4 * q)) & 15u;
        if (bits) {
            uint32_t rank = (uint32_t)(pre >> (16 * q)) & 0xFFFF;
            const uint32_t p = place + CSTAGE * q;  // its place in the tile
            uint32_t i = row_of(base + p, n, n_a, r0, r1);
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
                    uint32_t *o = stage + 3 * rank++;
                    o[0] = i;
                    o[1] = p + j - here + (n_a ? 0 : i + 1);  // B items count from 0
                    o[2] = v[q][j];
                }
            }
        }
        __syncwarp();
        const uint32_t words = to < cap ? 3 * (uint32_t)min((uint64_t)found, cap - to) : 0;
        uint32_t *o = out + 3 * to;
        for (uint32_t w = lane; w < words; w += 32) o[w] = stage[w];
        __syncwarp();
        to += found;
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

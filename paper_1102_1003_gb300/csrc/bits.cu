// Bit rows from CSR tidlists (the bitmap vertical representation, Sec. I-B).
//
// One warp writes one item's bits of a run of 16,384-transaction chunks (4,096 where
// there are few tasks, and then 512 bytes of shared memory, not 2 KiB): it finds
// the run's tids by two 32-way searches side by side (about log32 |S| dependent
// reads), then walks them in blocks of 256 (16-byte loads, the next block on its
// way), ORs a chunk's into 2 KiB of shared memory and stores its 64 blocks of 32
// bytes.  Every byte of the matrix is written once, so nothing is zeroed before,
// no global atomic is used and the lists' order is checked on the way.
// Bound: HBM, 4 bytes read per tid and 1 bit written per (item, transaction);
// short lists by the latency of the searches (hence runs), skewed families by
// the warps of full lists, one tid per bit, which end last (hence runs only
// where there are warps enough, and a block of its own for each).  Zipf n = 2,000,
// m = 10^6 (40 M tids, 250 MB of rows): 318 us with eight warps a block and 64-bit
// places, 287 with 32-bit ones, about 250 with one warp a block.
#include <algorithm>

#include "bits.cuh"

namespace bm {

constexpr int BW = 1;                                // warps per CTA: none waits for a neighbour with a longer list

// A longer list repeats tids; it is reported as not sorted without a look at it.  So
// places and searches take 32 bits.
constexpr uint32_t MAX_LIST = 1u << 30;

// One round of a 32-way search for the first index in [lo, hi) whose value is
// >= v, by the whole warp.  The result of all rounds is a function of the list
// and v alone, so neighbouring chunks agree on their border even when the list
// is not sorted.
__device__ __forceinline__ void search_round(const uint32_t *__restrict__ a, uint32_t &lo, uint32_t &hi, uint32_t v,
                                             uint32_t lane) {
    if (lo >= hi) return;  // done (warp-uniform): a further round could move the result of an unsorted list
    const uint32_t step = (hi - lo + 31) >> 5;  // (hi <= MAX_LIST: no overflow below)
    const uint32_t p = lo + lane * step + (step - 1);
    const bool below = p < hi && __ldg(&a[p]) < v;
    const uint32_t c = __popc(__ballot_sync(0xffffffffu, below));
    const uint32_t top = lo + c * step + (step - 1);  // the first probe not below, if c < 32
    lo = min(lo + c * step, hi);
    if (c < 32) hi = min(hi, top);
}

// BLOCK tids from place f of r, a 16-byte boundary, four per lane and load.  Places
// before `begin` hold `before` (the predecessor of the first), those from `end` on 0.
constexpr int BQ = 2;                  // loads in flight per lane and block
constexpr uint32_t BLOCK = 128 * BQ;
struct TidBlock {
    uint32_t x[BQ][4];
};
__device__ __forceinline__ void load_block(TidBlock &B, const uint32_t *__restrict__ r, uint32_t f, uint32_t begin,
                                           uint32_t end, uint32_t before, uint32_t lane) {
#pragma unroll
    for (int q = 0; q < BQ; q++) {
        const uint32_t i = f + 128u * q + 4u * lane;
        if (i >= begin && i + 4 <= end) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(r + i));
            B.x[q][0] = v.x; B.x[q][1] = v.y; B.x[q][2] = v.z; B.x[q][3] = v.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++) B.x[q][j] = i + j < begin ? before : i + j < end ? __ldg(&r[i + j]) : 0;
        }
    }
}

template <uint32_t CHUNK_KB>
__global__ void __launch_bounds__(32 * BW)
k_bits(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tids, uint32_t n, uint32_t m, BitsLayout L,
       uint32_t run, uint8_t *__restrict__ out, int *__restrict__ flags) {
    constexpr uint32_t CHUNK_BITS = CHUNK_KB * BITS_K;
    __shared__ __align__(16) uint32_t s_bits[BW][CHUNK_BITS / 32];
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t *bits = s_bits[threadIdx.x >> 5];
    uint4 *bits4 = reinterpret_cast<uint4 *>(bits);
    const uint32_t nchunk = (L.kblocks + CHUNK_KB - 1) / CHUNK_KB, nrun = (nchunk + run - 1) / run;
    const uint64_t tasks = (uint64_t)n * nrun, warps = (uint64_t)gridDim.x * BW;
    bool bad_tid = false, unsorted = false;
    // neighbouring warps: neighbouring items of the same chunks, whose 32-byte pieces share lines
    for (uint64_t w = blockIdx.x * (uint64_t)BW + (threadIdx.x >> 5); w < tasks; w += warps) {
        const uint32_t at = tasks >> 32 ? (uint32_t)(w / n) : (uint32_t)w / n, item = (uint32_t)(w - (uint64_t)at * n);
        const uint32_t c0 = at * run, c1 = min(c0 + run, nchunk);
        const uint64_t b = off[item], long_size = off[item + 1] - b;
        const uint32_t size = long_size <= MAX_LIST ? (uint32_t)long_size : 0;
        const uint32_t *a = tids + b;
        const uint32_t first = c0 * CHUNK_BITS, past = c1 * CHUNK_BITS;  // m <= 2^30: no overflow
        uint32_t e0 = 0, h0 = c0 ? size : 0, e1 = c1 == nchunk ? size : 0, h1 = size;
        while (e0 < h0 || e1 < h1) {
            search_round(a, e0, h0, first, lane);
            search_round(a, e1, h1, past, lane);
        }
        unsorted |= e1 < e0 || size != long_size;
        // places: from the 16-byte boundary at or before the run's first tid
        const uint32_t begin = (uint32_t)(reinterpret_cast<uintptr_t>(a + e0) >> 2) & 3u, end = begin + (e1 > e0 ? e1 - e0 : 0);
        const uint32_t *r = a + e0 - begin;
        uint32_t carry = e0 ? __ldg(&a[e0 - 1]) : 0;  // predecessor of the block's first tid
        uint32_t f = 0;                               // the block in hand; the one behind it is on its way
        TidBlock B, N;
        load_block(B, r, f, begin, end, carry, lane);
        load_block(N, r, f + BLOCK, begin, end, carry, lane);
        uint32_t b0 = 0;       // the block's first tid (carry: its last)
        bool fresh = true, plain = false;
        for (uint32_t c = c0; c < c1; c++) {
            const uint32_t x0 = c * CHUNK_BITS;
#pragma unroll
            for (uint32_t j = 0; j < CHUNK_BITS / 32 / 4; j += 32) bits4[j + lane] = make_uint4(0, 0, 0, 0);
            __syncwarp();
            for (;;) {
                if (fresh) {
                    // a new block.  plain: all places hold tids of the run, ascending and below m
                    const uint32_t last = __shfl_sync(0xffffffffu, B.x[BQ - 1][3], 31);
                    b0 = __shfl_sync(0xffffffffu, B.x[0][0], 0);
                    plain = f >= begin && f + BLOCK <= end && b0 >= first && last < past && last < m &&
                            ((f == 0 && e0 == 0) || carry < b0);
                    bool ok = true;
#pragma unroll
                    for (int q = 0; q < BQ; q++) {
                        const uint32_t up = __shfl_up_sync(0xffffffffu, B.x[q][3], 1);
                        const uint32_t head = q ? __shfl_sync(0xffffffffu, B.x[q ? q - 1 : 0][3], 31) : 0;
                        const uint32_t prev = lane ? up : head;
                        ok &= (q == 0 && lane == 0) || prev < B.x[q][0];
                        ok &= B.x[q][0] < B.x[q][1] && B.x[q][1] < B.x[q][2] && B.x[q][2] < B.x[q][3];
                    }
                    plain = plain && __all_sync(0xffffffffu, ok);
                    if (!plain) {  // place by place
#pragma unroll
                        for (int q = 0; q < BQ; q++) {
                            const uint32_t i = f + 128u * q + 4u * lane;
                            uint32_t prev = __shfl_up_sync(0xffffffffu, B.x[q][3], 1);
                            if (lane == 0) prev = carry;
#pragma unroll
                            for (int j = 0; j < 4; j++) {
                                const uint32_t y = B.x[q][j];
                                if (i + j >= begin && i + j < end) {
                                    // (the list's first tid has no predecessor)
                                    unsorted |= ((e0 || i + j != begin) && !(prev < y)) || y < first || y >= past;
                                    bad_tid |= y >= m;
                                }
                                prev = y;
                            }
                            carry = __shfl_sync(0xffffffffu, B.x[q][3], 31);
                        }
                    }
                    carry = last;
                }
#pragma unroll
                for (int q = 0; q < BQ; q++) {
                    const uint32_t i = f + 128u * q + 4u * lane;
                    uint32_t word = 0, mask = 0;  // bits of one word are set together
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const uint32_t y = B.x[q][j];
                        if (y - x0 < CHUNK_BITS && (plain || (y < m && i + j >= begin && i + j < end))) {
                            const uint32_t v = (y - x0) >> 5;
                            if (v != word && mask) {
                                atomicOr(&bits[word], mask);
                                mask = 0;
                            }
                            word = v;
                            mask |= 1u << (y & 31u);
                        }
                    }
                    if (mask) atomicOr(&bits[word], mask);
                }
                // the chunk goes on in the next block if this one's last tid (carry) lies before its end
                fresh = f + BLOCK < end && carry < x0 + CHUNK_BITS;
                if (!fresh) break;
                f += BLOCK;
                B = N;
                load_block(N, r, f + BLOCK, begin, end, carry, lane);
            }
            __syncwarp();
            uint8_t *row = out + item * L.row_stride;
#pragma unroll
            for (uint32_t j = 0; j < CHUNK_KB * 2; j += 32) {
                const uint32_t i = j + lane, kb = c * CHUNK_KB + (i >> 1);
                if (kb < L.kblocks) *reinterpret_cast<uint4 *>(row + kb * L.kb_stride + 16u * (i & 1u)) = bits4[i];
            }
            __syncwarp();
        }
        unsorted |= f + BLOCK < end;  // (a sorted run ends with its last block)
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

// Blocks per chunk.  Fewer chunks than FEW_TASKS (two warps for each that the chip holds): a quarter of that, as
// the time is that of a full list's chunk (triples of n = 1,000, m = 100,000
// with full lists: the pass 1572 -> 1542 us).
constexpr uint32_t CHUNK_KB = 64;
constexpr uint64_t FEW_TASKS = 152 * 32 * 2;

template <uint32_t KB>
static void launch_bits(const uint64_t *d_off, const uint32_t *d_tids, uint32_t n, uint32_t m, const BitsLayout &L,
                        uint32_t run, uint8_t *d_bits, int *d_flags, cudaStream_t st) {
    const uint32_t nchunk = (L.kblocks + KB - 1) / KB;
    const uint64_t tasks = (uint64_t)n * ((nchunk + run - 1) / run);
    const unsigned grid = (unsigned)std::min<uint64_t>((tasks + BW - 1) / BW, 1u << 20);
    k_bits<KB><<<grid, 32 * BW, 0, st>>>(d_off, d_tids, n, m, L, run, d_bits, d_flags);
}

void enqueue_bits(const uint64_t *d_off, const uint32_t *d_tids, uint32_t n, uint32_t m, const BitsLayout &L,
                  uint8_t *d_bits, int *d_flags, bool sorted_only, cudaStream_t st) {
    if (!n) return;
    const uint32_t nchunk = (L.kblocks + CHUNK_KB - 1) / CHUNK_KB;
    if ((uint64_t)n * nchunk < FEW_TASKS)
        launch_bits<CHUNK_KB / 4>(d_off, d_tids, n, m, L, 1, d_bits, d_flags, st);
    else  // chunks per warp: about 200,000 warps (many rounds of the chip) before a warp takes several,
          // which saves it their searches
        launch_bits<CHUNK_KB>(d_off, d_tids, n, m, L,
                              (uint32_t)std::min<uint64_t>(16, std::max<uint64_t>(1, (uint64_t)n * nchunk / 200000)), d_bits,
                              d_flags, st);
    BM_CHECK_LAUNCH();
    if (!sorted_only) {
        k_bits_unsorted<<<dim3(8, std::min<uint32_t>(n, 128u)), 256, 0, st>>>(d_off, d_tids, n, m, L, d_bits, d_flags);
        BM_CHECK_LAUNCH();
    }
}

bool take_bits(BmBuf *buf, uint64_t bytes, uint64_t supports) {
    if (bytes > (64ull << 20)) {
        const uint64_t available = device_available();
        if (available < supports || bytes > (available - supports) / 2) return false;
    }
    try {
        buf->alloc(bytes);
    } catch (const Error &e) {
        if (e.code != BATMAP_ERR_NOMEM) throw;
        return false;  // not an error of this call: the BatMap routes need no bits
    }
    return true;
}

// ---- k-way supports ------------------------------------------------------------
//
// A group of W warps takes G consecutive queries.  The queries of a candidate
// list are in lexicographic order, so most share all ids but the last: their
// common AND is formed once per 16-byte chunk, and each query costs one load,
// four ANDs and four popcounts per chunk.  Queries that differ earlier go one by
// one.  Rows come from L2 (12.5 MB at m = 100,000, n = 1,000) and, for the shared
// ones, from L1; popcount issues at 16 per clock and SM, so 511,714 triples of
// 3,128 words take at least 0.32 ms, and their rows 6.4 GB of L2 reads; measured
// 0.46 ms with three blocks a multiprocessor (67 registers), 0.43 with four.
template <int K, int G, int W>
__global__ void __launch_bounds__(256, 4) k_bits_support(const uint4 *__restrict__ bits, uint32_t chunks,
                                                      const uint32_t *__restrict__ items, uint64_t nq,
                                                      uint32_t *__restrict__ out) {
    const uint32_t t = threadIdx.x % (32 * W);
    const uint64_t groups = (uint64_t)gridDim.x * (8 / W);
    __shared__ uint32_t s_sum[8];
    for (uint64_t q0 = (blockIdx.x * (uint64_t)(8 / W) + threadIdx.x / (32 * W)) * G; q0 < nq; q0 += groups * G) {
        const uint32_t gn = (uint32_t)min((uint64_t)G, nq - q0);
        const uint32_t *it = items + q0 * K;
        bool same = true;
        for (uint32_t j = 1; j < gn; j++)
#pragma unroll
            for (int p = 0; p < K - 1; p++) same &= __ldg(&it[j * K + p]) == __ldg(&it[p]);
        uint32_t cnt[G];
#pragma unroll
        for (int j = 0; j < G; j++) cnt[j] = 0;
        if (same) {
            const uint4 *pre[K], *last[G];
#pragma unroll
            for (int p = 0; p < K - 1; p++) pre[p] = bits + (uint64_t)__ldg(&it[p]) * chunks;
#pragma unroll
            for (int j = 0; j < G; j++) last[j] = bits + (uint64_t)__ldg(&it[((uint32_t)j < gn ? j : 0) * K + K - 1]) * chunks;
            for (uint32_t c = t; c < chunks; c += 32 * W) {
                uint4 v = make_uint4(~0u, ~0u, ~0u, ~0u), y[G];
#pragma unroll
                for (int j = 0; j < G; j++) y[j] = __ldg(last[j] + c);
#pragma unroll
                for (int p = 0; p < K - 1; p++) {
                    const uint4 x = __ldg(pre[p] + c);
                    v.x &= x.x; v.y &= x.y; v.z &= x.z; v.w &= x.w;
                }
#pragma unroll
                for (int j = 0; j < G; j++)
                    cnt[j] += __popc(v.x & y[j].x) + __popc(v.y & y[j].y) + __popc(v.z & y[j].z) + __popc(v.w & y[j].w);
            }
        } else {
#pragma unroll
            for (int j = 0; j < G; j++) {
                if ((uint32_t)j >= gn) break;
                const uint4 *row[K];
#pragma unroll
                for (int p = 0; p < K; p++) row[p] = bits + (uint64_t)__ldg(&it[j * K + p]) * chunks;
#pragma unroll 2
                for (uint32_t c = t; c < chunks; c += 32 * W) {
                    uint4 v = __ldg(row[0] + c);
#pragma unroll
                    for (int p = 1; p < K; p++) {
                        const uint4 x = __ldg(row[p] + c);
                        v.x &= x.x; v.y &= x.y; v.z &= x.z; v.w &= x.w;
                    }
                    cnt[j] += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < G; j++) {
            const uint32_t sum = __reduce_add_sync(0xffffffffu, cnt[j]);
            if (W == 1) {
                if (t == 0 && (uint32_t)j < gn) out[q0 + j] = sum;
            } else {  // G == 1: one query per block
                if ((threadIdx.x & 31u) == 0) s_sum[threadIdx.x >> 5] = sum;
                __syncthreads();
                if (threadIdx.x == 0) {
                    uint32_t all = 0;
                    for (int w = 0; w < 8; w++) all += s_sum[w];
                    out[q0] = all;
                }
                __syncthreads();
            }
        }
    }
}

template <int K>
static void launch_bits_support(const uint4 *bits, uint32_t chunks, const uint32_t *items, uint64_t nq, uint32_t *out,
                                cudaStream_t st) {
    // few queries: a block each, so that one long row does not wait on one warp
    constexpr uint64_t FEW = 152 * 8;
    if (nq <= FEW) {
        k_bits_support<K, 1, 8><<<(unsigned)nq, 256, 0, st>>>(bits, chunks, items, nq, out);
    } else {
        constexpr int G = K == 1 ? 1 : K == 4 ? 4 : 8;
        const uint64_t blocks = (nq + 8ull * G - 1) / (8ull * G);
        k_bits_support<K, G, 1><<<(unsigned)std::min<uint64_t>(blocks, 1u << 20), 256, 0, st>>>(bits, chunks, items, nq, out);
    }
    BM_CHECK_LAUNCH();
}

void enqueue_bits_support(const uint8_t *d_bits, uint32_t kblocks, uint32_t k, const uint32_t *d_items, uint64_t nq,
                          uint32_t *d_support, cudaStream_t st) {
    if (!nq) return;
    const uint4 *bits = reinterpret_cast<const uint4 *>(d_bits);
    const uint32_t chunks = kblocks * 2;
    if (k == 1) launch_bits_support<1>(bits, chunks, d_items, nq, d_support, st);
    if (k == 2) launch_bits_support<2>(bits, chunks, d_items, nq, d_support, st);
    if (k == 3) launch_bits_support<3>(bits, chunks, d_items, nq, d_support, st);
    if (k == 4) launch_bits_support<4>(bits, chunks, d_items, nq, d_support, st);
}

}  // namespace bm

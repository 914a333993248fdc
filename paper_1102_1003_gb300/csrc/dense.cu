// Supports of all pairs as the dense boolean contraction C = M M^T over bit
// rows, M in {0,1}^(n x m) (items x transactions; Sec. I-A / Sec. I-B: the
// bitmap vertical representation, AND + popcount), on the 5th-generation
// tensor cores.  It serves pair_support_dense and the pair calls on built sets
// whose estimated time is lower this way than by the BatMap scan.
//
//   * M stays packed in HBM, one bit per (item, transaction), in blocks of 256
//     transactions, each block's rows of 32 bytes one after the other, so the
//     rows of a tile are one contiguous bulk copy per block;
//   * a CTA computes 256 rows x 240 columns as two 128 x 240 tiles that share
//     their B operand; per block of 256 transactions one bulk copy each brings
//     the bits of the A and the B rows (15.5 KiB, 2-stage ring), two groups of
//     eight expander warps, a block each in turn, turn them into e2m1 {0, 1} nibbles (1.0 = 0x2) in the
//     128-byte-swizzled layout the MMA reads (62 KiB, 3-stage ring) and publish
//     each stage after a proxy fence;
//   * one thread issues tcgen05.mma.cta_group::1.kind::mxf4 (M = 128, N = 240,
//     K = 64, every block scale 2^0) into two FP32 accumulators; with the scales
//     they fill the 512 columns of tensor memory (hence 240 columns, not 256);
//   * all expander warps read the accumulators with tcgen05.ld, transpose 32 x 32
//     pieces through shared memory and store (or, for a split K, add) rows of
//     32 consecutive supports.
//
// Exactness: every product is exactly 0 or 1 and every partial sum an integer
// of at most 2^24 (a unit spans at most 2^24 transactions), which the FP32
// accumulator represents exactly; partial sums of a split K are added as
// integers.  INT8 MMA (kind::i8) is not available on sm_103a.
//
// What bounds it: the MMA pipe, 173 clk per 128 x 240 x 64 with stale operands
// (7.1 PFLOP/s), which the nibble stores slow to 217 (5.7): m = 2^22, n = 8,192
// takes 54.4 ms, 43.3 without the stores.  Pairs of CTAs (cta_group::2), which
// expand and read each B row once for two, were no faster (54.5 ms): the bytes
// through shared memory (105 of 128 per clk here, 76 there) are not what counts.
// One group of sixteen warps, a row per thread: 54.7 ms, and 0.36 instead of
// 0.34 ms on short K (m = 25,000, n = 8,000).  e4m3 operands (kind::f8f6f4,
// K = 32): 92 ms.
//
// Every mbarrier wait is bounded; on timeout the kernel records an error
// flag, stops issuing work, waits (bounded) for what it issued, frees its
// tensor memory and returns.  A test hook (batmap_test_dense_timeout) runs
// one launch whose producer issues no loads and whose waits are short, so
// that every wait gives up with nothing in flight.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>

#include "bits.cuh"
#include "common.cuh"
#include "compare.cuh"
#include "scan.cuh"

namespace bm {

void enqueue_threshold(const uint32_t *C, uint64_t n, uint32_t s, uint32_t *d_pairs, uint64_t cap,
                       DevBuf<uint64_t> *state, uint64_t *d_total, cudaStream_t st);

namespace dense {

constexpr int BM = 128, BN = MM_COLS, STAGES = 3, SB = 2;
constexpr int ROWS = 2 * BM + BN;                  // rows of a stage: A0, A1, B
constexpr uint32_t ROW_BYTES = BITS_K / 2;         // 128: 256 e2m1 values
constexpr uint32_t A_BYTES = BM * ROW_BYTES;       // 16 KiB per A tile (two per stage)
constexpr uint32_t STAGE_BYTES = ROWS * ROW_BYTES; // 62 KiB
constexpr uint32_t BIT_ROW = BITS_K / 8;           // 32 bytes of bits per row and block
constexpr uint32_t BITS_STAGE = ROWS * BIT_ROW;    // 15.5 KiB
constexpr int MMA_PER_STAGE = BITS_K / 64;         // K = 64 per MMA: 32 bytes of a row
constexpr uint32_t TMEM_COLS = 512;                // accumulators at 0 and ACC1, scales at SFA, SFB
constexpr uint32_t SFA = 240, SFB = 248, ACC1 = 256;
constexpr int NG = 2, RPT = 2;                     // expander groups, a step each in turn; rows per thread
constexpr int XW = (ROWS + 32 * RPT - 1) / (32 * RPT);  // warps of a group
constexpr int EW = NG * XW;                        // warps 2 .. 17: expanders, then the epilogue
constexpr int THREADS = 64 + 32 * EW;              // warp 0 copies, warp 1 MMA
constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + (size_t)SB * BITS_STAGE + 1024 /*align*/ + 256;
static_assert(SMEM <= 232448, "shared memory of one CTA");
static_assert(A_BYTES % 1024 == 0 && STAGE_BYTES % 1024 == 0, "swizzle atoms");
static_assert(EW * 32 * 33 * 4 <= STAGES * STAGE_BYTES && EW % 4 == 0, "epilogue staging fits the ring");
// a group waits for every use of its bits stages, a parity at a time; of the nibble stages its waits
// are at most NG <= STAGES steps apart, so a parity never stands for an older use
static_assert(SB % NG == 0 && NG <= STAGES, "barrier phases");
constexpr uint32_t SPIN_LIMIT = 1u << 26;          // bounded waits (tens of ms per wait)

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait for the phase with the given parity (at most `limit` polls);
// false on timeout.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t limit) {
    for (uint32_t it = 0; it < limit; it++) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// Contiguous copy; both addresses and the size are multiples of 16 bytes.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile stored with the
// 128-byte swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);  // start address
    d |= (uint64_t)1 << 16;                    // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;          // stride byte offset: 8 rows x 128 B
    d |= (uint64_t)1 << 46;                    // descriptor version
    d |= (uint64_t)2 << 61;                    // 128-byte swizzle
    return d;
}

// Instruction descriptor of kind::mxf4: A = B = E2M1 (1), both K-major, scales UE8M0, M = 128,
// N = 240, dense K = 64, scale data ids 0.
constexpr uint32_t IDESC = (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | (1u << 23) |
                           ((uint32_t)(BM >> 4) << 24);

__device__ __forceinline__ void umma_mxf4(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t sfa, uint32_t sfb,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%6], p;\n}\n"
        ::"r"(tmem_d), "l"(da), "l"(db), "r"(IDESC), "r"(accumulate), "r"(sfa), "r"(sfb));
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// 32 bits to 32 e2m1 nibbles, a set bit to 1.0 (0x2).  Output word j holds bits
// j, j + 4, .., j + 28: a fixed order of the K values, the same for both
// operands, which a contraction does not see.
__device__ __forceinline__ uint4 expand32(uint32_t w) {
    constexpr uint32_t ONE = 0x22222222u;
    return make_uint4((w << 1) & ONE, w & ONE, (w >> 1) & ONE, (w >> 2) & ONE);
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Persistent: one CTA per SM pulls units until the queue is empty.
__global__ void __launch_bounds__(THREADS, 1)
k_contract(const MmView *__restrict__ views, const MmView one, const MmUnit *__restrict__ units, uint32_t count,
           uint32_t *__restrict__ state, uint32_t spin, uint32_t no_loads, unsigned long long *stamps) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *bits = smem + STAGES * STAGE_BYTES;
    uint64_t *bars = reinterpret_cast<uint64_t *>(bits + SB * BITS_STAGE);
    // bars: bits full (bulk copies), bits empty (expanders), nibbles full (expanders), nibbles
    // empty (MMA commit), accumulators ready (MMA commit)
    constexpr int BF = 0, BE = SB, YF = 2 * SB, YE = 2 * SB + STAGES, ACC = 2 * SB + 2 * STAGES;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + ACC + 1);
    __shared__ volatile int s_abort;
    __shared__ uint32_t s_unit;
    int *err = reinterpret_cast<int *>(state + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (stamps && threadIdx.x == 0) atomicMin(&stamps[0], (unsigned long long)global_ns());
    if (threadIdx.x == 0) {
        s_abort = 0;
        s_unit = atomicAdd(&state[0], 1u);
        for (int i = 0; i <= ACC; i++)
            mbar_init(smem_addr(&bars[i]), (i >= BE && i < BE + SB) || (i >= YF && i < YF + STAGES) ? XW : 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_addr(tmem_slot)), "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    if (warp >= 2 && warp < 6) {
        // every block scale of both operands is 2^0 (UE8M0 0x7F): 16 columns of all 128 lanes
        const uint32_t q = warp & 3, one = 0x7F7F7F7Fu;
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};"
            ::"r"(tmem + ((q * 32u) << 16) + SFA), "r"(one)
            : "memory");
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    uint32_t step0 = 0, round = 0;  // K steps and units done: the rings' and the accumulators' phases
    for (uint32_t u = s_unit; u < count; round++) {
        const MmUnit U = units[u];
        const MmView V = views ? views[U.inst] : one;
        const uint32_t nk = U.kb1 - U.kb0;
        const uint32_t clim = min(U.c0 + (uint32_t)BN, V.n);  // columns [c0, clim)
        // does the second A tile hold a pair that is reported?
        const bool half1 = V.n_a ? U.r0 + BM < V.n_a : U.r0 + BM + 1 < clim;
        const uint32_t ra = min(half1 ? 2u * BM : (uint32_t)BM, V.n - U.r0), rb = clim - U.c0;

        if (warp == 0 && lane == 0) {
            // copies of the packed bits (no_loads: the timeout test issues nothing); rows past the
            // matrix keep old bits: they only reach supports that are not stored
            uint32_t it = 0;
            for (; it < nk && !s_abort && !no_loads; it++) {
                const uint32_t g = step0 + it, sb = g % SB, use = g / SB;
                if (use > 0 && !mbar_wait(smem_addr(&bars[BE + sb]), (use - 1) & 1, spin)) {
                    atomicExch(err, 1);
                    s_abort = 1;
                    break;
                }
                const uint32_t full = smem_addr(&bars[BF + sb]);
                const uint8_t *src = V.bits + (uint64_t)(U.kb0 + it) * V.n * BIT_ROW;
                uint8_t *dst = bits + sb * BITS_STAGE;
                mbar_expect_tx(full, (ra + rb) * BIT_ROW);
                bulk_load(smem_addr(dst), src + (uint64_t)U.r0 * BIT_ROW, ra * BIT_ROW, full);
                bulk_load(smem_addr(dst + 2 * BM * BIT_ROW), src + (uint64_t)U.c0 * BIT_ROW, rb * BIT_ROW, full);
            }
            if (s_abort) {
                // wait (bounded) for the last copies issued into every bits stage
                for (uint32_t b = 0; b < (uint32_t)SB && b < it; b++) {
                    const uint32_t g = step0 + it - 1 - b;
                    mbar_wait(smem_addr(&bars[BF + g % SB]), (g / SB) & 1, spin);
                }
            }
        } else if (warp == 1 && lane == 0) {
            // MMA issuer
            for (uint32_t it = 0; it < nk; it++) {
                const uint32_t g = step0 + it, st = g % STAGES;
                if (s_abort || !mbar_wait(smem_addr(&bars[YF + st]), (g / STAGES) & 1, spin)) {
                    atomicExch(err, 1);
                    s_abort = 1;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t a0 = smem_addr(smem + st * STAGE_BYTES);
                const uint64_t da0 = smem_desc(a0), da1 = smem_desc(a0 + A_BYTES), db = smem_desc(a0 + 2 * A_BYTES);
#pragma unroll
                for (int k = 0; k < MMA_PER_STAGE; k++) {
                    // advance 64 nibbles = 32 bytes along K inside the swizzled 128-byte rows
                    const uint32_t acc = (it > 0 || k > 0) ? 1u : 0u;
                    umma_mxf4(tmem, da0 + (uint64_t)(k * 2), db + (uint64_t)(k * 2), tmem + SFA, tmem + SFB, acc);
                    if (half1)
                        umma_mxf4(tmem + ACC1, da1 + (uint64_t)(k * 2), db + (uint64_t)(k * 2), tmem + SFA, tmem + SFB,
                                  acc);
                }
                umma_commit(smem_addr(&bars[YE + st]));  // frees the stage when the MMAs have read it
            }
            umma_commit(smem_addr(&bars[ACC]));  // accumulators ready (or nothing issued)
        } else if (warp >= 2) {
            // expanders: a thread owns rows t0 + 32 XW r (A0 0..127, A1 128..255, B 256..495); row r of a
            // stage starts at r * 128, 16-byte chunk c at c ^ (r & 7)
            const uint32_t grp = (uint32_t)(warp - 2) / XW, t0 = (uint32_t)((warp - 2) % XW) * 32u + lane;
            for (uint32_t it = 0; it < nk; it++) {
                const uint32_t g = step0 + it, sb = g % SB, st = g % STAGES;
                if (g % NG != grp) continue;
                bool ok = !s_abort && mbar_wait(smem_addr(&bars[BF + sb]), (g / SB) & 1, spin);
                if (ok && g >= (uint32_t)STAGES)
                    ok = mbar_wait(smem_addr(&bars[YE + st]), ((g / STAGES) - 1) & 1, spin);
                if (!ok) {
                    atomicExch(err, 1);
                    s_abort = 1;
                    break;
                }
#pragma unroll
                for (int r = 0; r < RPT; r++) {
                    const uint32_t t = t0 + (uint32_t)(32 * XW * r);
                    if (t >= (uint32_t)ROWS || (!half1 && t >= (uint32_t)BM && t < 2u * BM)) continue;
                    const uint4 *src = reinterpret_cast<const uint4 *>(bits + sb * BITS_STAGE + t * BIT_ROW);
                    uint8_t *row = smem + st * STAGE_BYTES + t * ROW_BYTES;
                    const uint4 w0 = src[0], w1 = src[1];
                    const uint32_t ws[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
                    for (int c = 0; c < 8; c++)
                        *reinterpret_cast<uint4 *>(row + ((((uint32_t)c) ^ (t & 7u)) << 4)) = expand32(ws[c]);
                }
                // generic-proxy writes become visible to the tensor core's reads
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(smem_addr(&bars[YF + st]));
                    mbar_arrive(smem_addr(&bars[BE + sb]));
                }
            }
            // epilogue: TMEM lanes 32 (warp mod 4) .. +31 hold tile rows of that quarter; the four warps
            // of a quarter share its 2 x 8 pieces of 32 columns
            const uint32_t q = warp & 3, gq = (uint32_t)(warp - 2) >> 2;
            bool ready = false;
            for (int rep = 0; rep < 16 && !ready; rep++) ready = mbar_wait(smem_addr(&bars[ACC]), round & 1, spin);
            if (!ready) {
                atomicExch(err, 1);
                s_abort = 1;
            } else if (!s_abort) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                uint32_t *stg = reinterpret_cast<uint32_t *>(smem) + (warp - 2) * (32 * 33);  // the MMAs are done
                const uint64_t nn = V.n;
#pragma unroll 1
                for (uint32_t p = gq; p < 16; p += EW / 4) {
                    const uint32_t h = p >> 3, c0 = (p & 7u) * 32u;
                    if (h && !half1) break;
                    const uint32_t gi0 = U.r0 + h * BM + q * 32u, gj = U.c0 + c0 + (uint32_t)lane;
                    const uint32_t ilim = V.n_a ? V.n_a : min(clim, U.c0 + c0 + 32u) - 1u;  // rows < ilim hold a pair
                    if (gi0 >= ilim || U.c0 + c0 >= clim) continue;                          // warp-uniform
                    uint32_t v[32];
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
                          "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),
                          "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
                          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]),
                          "=r"(v[31])
                        : "r"(tmem + ((q * 32u) << 16) + h * ACC1 + c0));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int c = 0; c < 32; c++) stg[lane * 33 + c] = __float2uint_rn(__uint_as_float(v[c]));
                    __syncwarp();
                    const bool col = gj < clim;
                    const uint32_t rows = min(32u, ilim - gi0);
                    // supports of row i start at rb: triangle i n - i (i + 1) / 2 - i - 1, rectangle i n_b - n_a
                    uint64_t at = V.n_a ? (uint64_t)gi0 * (nn - V.n_a) - V.n_a
                                        : (uint64_t)gi0 * nn - (uint64_t)gi0 * (gi0 + 1ull) / 2 - gi0 - 1;
                    for (uint32_t r = 0; r < rows; r++) {
                        const uint32_t gi = gi0 + r, x = stg[r * 33 + lane];
                        if (col && (V.n_a || gi < gj)) {
                            if (!U.add) V.C[at + gj] = x;
                            else if (x) atomicAdd(&V.C[at + gj], x);
                        }
                        at += V.n_a ? nn - V.n_a : nn - gi - 2;
                    }
                    __syncwarp();
                }
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();  // accumulators and stages are free again
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (s_abort) break;
        if (threadIdx.x == 0) s_unit = atomicAdd(&state[0], 1u);
        step0 += nk;
        __syncthreads();
        u = s_unit;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
    }
    if (stamps && threadIdx.x == 0) atomicMax(&stamps[1], (unsigned long long)global_ns());
}

}  // namespace dense

// ---- units -----------------------------------------------------------------------

// Seconds of one K block of a 256 x 240 unit and of a unit's fill and epilogue.
constexpr double MM_STEP_S = 0.84e-6, MM_UNIT_S = 8e-6, MM_LAUNCH_S = 10e-6;

// Tiles holding a reported pair: row blocks of 256 from 0, column blocks of 240 from the first
// column (cross: family B).
template <typename F>
static void each_tile(uint32_t n, uint32_t n_a, F &&f) {
    const uint32_t rows = n_a ? n_a : n, col0 = n_a;
    for (uint32_t c0 = col0; c0 < n; c0 += MM_COLS) {
        const uint32_t clim = std::min<uint64_t>((uint64_t)c0 + MM_COLS, n);
        for (uint32_t r0 = 0; r0 < rows && (n_a || r0 + 1 < clim); r0 += MM_ROWS) f(r0, c0);
    }
}

static uint64_t count_tiles(uint32_t n, uint32_t n_a) {
    if (n_a) return (uint64_t)((n_a + MM_ROWS - 1) / MM_ROWS) * ((n - n_a + MM_COLS - 1) / MM_COLS);
    uint64_t k = 0;
    for (uint64_t c0 = 0; c0 < n; c0 += MM_COLS) {
        const uint64_t clim = std::min<uint64_t>(c0 + MM_COLS, n);
        if (clim > 1) k += (clim - 1 + MM_ROWS - 1) / MM_ROWS;
    }
    return k;
}

// Pieces of the K blocks of each of T equal tiles: the waves of equal units over the SMs that end
// first, epilogues included; a piece spans at most 2^24 transactions (exact FP32 sums) and, when
// split for balance, at least 4 blocks.
static uint32_t k_pieces(uint64_t T, uint32_t kblocks, double sms) {
    const uint32_t least = std::max<uint32_t>(1, (uint32_t)((kblocks + 65535ull) / 65536));
    uint32_t best = least;
    double best_t = INFINITY;
    for (uint32_t k = least; k <= least + 64 && (k == least || 4ull * k <= kblocks); k++) {
        const double waves = std::ceil((double)T * k / sms);
        const double t = waves * (std::ceil((double)kblocks / k) * MM_STEP_S + MM_UNIT_S);
        if (t < best_t * 0.99) {
            best_t = t;
            best = k;
        }
    }
    return best;
}

double contract_seconds(uint32_t n, uint32_t n_a, uint32_t kblocks) {
    const uint64_t T = count_tiles(n, n_a);
    const uint32_t k = k_pieces(T, kblocks, device_sms());
    return MM_LAUNCH_S + std::ceil((double)T * k / device_sms()) *
                             (std::ceil((double)kblocks / k) * MM_STEP_S + MM_UNIT_S);
}

bool contract_units(uint32_t n, uint32_t n_a, uint32_t kblocks, uint32_t inst, double others,
                    std::vector<MmUnit> *out) {
    const uint64_t T = count_tiles(n, n_a);
    uint32_t k = k_pieces(T, kblocks, device_sms());
    if (others > 0.0) {
        // one of several instances: units no longer than an eighth of an SM's share of the launch
        const double tile_s = kblocks * MM_STEP_S, share = (others + (double)T * tile_s / device_sms()) / 8;
        const uint32_t least = std::max<uint32_t>(1, (uint32_t)((kblocks + 65535ull) / 65536));
        k = std::max<uint32_t>(least, (uint32_t)std::min(std::ceil(tile_s / std::max(share, 4 * MM_UNIT_S)),
                                                        std::max(1.0, kblocks / 4.0)));
    }
    each_tile(n, n_a, [&](uint32_t r0, uint32_t c0) {
        for (uint32_t p = 0; p < k; p++)
            out->push_back({r0, c0, (uint32_t)((uint64_t)kblocks * p / k), (uint32_t)((uint64_t)kblocks * (p + 1) / k),
                            inst, k > 1 ? 1u : 0u, {0, 0}});
    });
    return k > 1;
}

void prepare_contract() {
    static std::once_flag once;
    std::call_once(once, [] {
        BM_CUDA(cudaFuncSetAttribute(dense::k_contract, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)dense::SMEM));
    });
}

void launch_contract(const MmView *d_views, const MmView &one, const MmUnit *d_units, uint32_t count,
                     uint32_t *d_state, cudaStream_t st, unsigned long long *d_stamps, uint32_t test_spin) {
    if (!count) return;
    prepare_contract();
    dense::k_contract<<<std::min<uint32_t>(count, (uint32_t)device_sms()), dense::THREADS, dense::SMEM, st>>>(
        d_views, one, d_units, count, d_state, test_spin ? test_spin : dense::SPIN_LIMIT, test_spin ? 1u : 0u, d_stamps);
    BM_CHECK_LAUNCH();
}

// ---- built sets ----------------------------------------------------------------------
//
// A set's supports come from its bit rows where that is estimated faster than
// the BatMap scan, the bits' build included.  The scan costs four integer
// instructions per 32-bit word pair: 7e12 word pairs/s on large instances
// (9.5 ms for the 6.6e10 of the m = 10^6, n = 2,000 Zipf workload after the probe
// route), and about 40 us of latency on the smallest; the contraction 256 x 240
// pairs x 256 transactions per SM in MM_STEP_S.  BatMaps are at least m / 42
// bytes wide, so the scan wins only where tiles are mostly padding: few items
// over many transactions.  A caller who sets tile, shape_mask or probe_log asks
// for a BatMap route and gets it.  The bits are left out (and the scan taken)
// where they would take more than half of the memory that is free beside the supports.
// Measured where the rule switches (n = 2 to 300, m = 5,000 to 2^26, 184 builds with their
// supports): where it takes the contraction that is never the slower route.
constexpr double SCAN_WORD_PAIRS_PER_S = 7e12, SCAN_MIN_S = 40e-6, BITS_BYTES_PER_S = 4e12;

void plan_contract(batmap_set *S, const uint64_t *d_off, const uint32_t *d_tids, int *d_flags, bool sorted_only,
                   cudaStream_t st) {
    const batmap_params &P = S->params;
    S->contract = false;
    if (S->skip_schedule || P.tile || P.shape_mask || P.probe_log || !S->npairs() || !S->n_elements) return;
    const BitsLayout L = bits_block_major(S->n, S->m);
    const uint64_t bytes = L.kb_stride * L.kblocks;
    const double bits_s = ((double)bytes + 4.0 * (double)S->n_elements) / BITS_BYTES_PER_S;
    if (bits_s + contract_seconds(S->n, S->n_a, L.kblocks) > SCAN_MIN_S + S->word_pairs / SCAN_WORD_PAIRS_PER_S) return;
    if (!take_bits(&S->d_bits, bytes, S->npairs() * sizeof(uint32_t))) return;
    std::vector<MmUnit> units;
    S->mm_add = contract_units(S->n, S->n_a, L.kblocks, 0, 0.0, &units);
    S->mm_count = (uint32_t)units.size();
    S->kblocks = L.kblocks;
    S->d_mm.alloc(64 + units.size() * sizeof(MmUnit));
    BM_CUDA(cudaMemcpyAsync(S->d_mm.p + 64, units.data(), units.size() * sizeof(MmUnit), cudaMemcpyHostToDevice,
                            st));
    enqueue_bits(d_off, d_tids, S->n, S->m, L, S->d_bits.p, d_flags, sorted_only, st);
    S->contract = true;
}

MmView contract_view(const batmap_set *S, uint32_t *C) { return MmView{S->d_bits.p, C, S->n, S->n_a}; }

void enqueue_contract(batmap_set *S, uint32_t *C, cudaStream_t st) {
    if (S->mm_add) BM_CUDA(cudaMemsetAsync(C, 0, S->npairs() * sizeof(uint32_t), st));
    BM_CUDA(cudaMemsetAsync(S->d_mm.p, 0, 64, st));
    launch_contract(nullptr, contract_view(S, C), reinterpret_cast<const MmUnit *>(S->d_mm.p + 64), S->mm_count,
                    reinterpret_cast<uint32_t *>(S->d_mm.p), st);
}

// ---- pair_support_dense ------------------------------------------------------------

// Workspace kept across calls (bit rows, supports, units, scratch).
struct DenseWork {
    DevBuf<uint8_t> bits;
    DevBuf<uint32_t> C;
    DevBuf<MmUnit> units;
    DevBuf<uint32_t> state;   // queue counter, timeout flag, bit flags (tid >= m, unsorted)
    DevBuf<uint64_t> blocksums, total;
    PhaseEvents ev;
    batmap_timing timing{};
};

static std::mutex g_dense_mu;
static DenseWork *g_dense = nullptr;
static std::atomic<uint32_t> g_dense_timeout_test{0};  // one-shot spin limit of the timeout test

void set_dense_timeout_test(uint32_t spin_limit) { g_dense_timeout_test.store(spin_limit); }

void release_dense_workspace() {
    std::lock_guard<std::mutex> lock(g_dense_mu);
    delete g_dense;
    g_dense = nullptr;
}

void run_dense(uint32_t m, uint32_t n, const uint64_t *d_off, const uint32_t *d_tids, uint32_t s,
               uint32_t *d_pairs, uint64_t cap, uint64_t *n_out, uint32_t *d_full, batmap_timing *tout,
               cudaStream_t st) {
    BM_REQUIRE(n_out, BATMAP_ERR_ARG, "n_out is NULL");
    BM_REQUIRE(cap == 0 || d_pairs, BATMAP_ERR_ARG, "d_pairs is NULL with cap > 0");
    BM_REQUIRE(m >= 1 && m <= (1u << 24), BATMAP_ERR_ARG, "dense path needs 1 <= m <= 2^24 (exact FP32 sums)");
    BM_REQUIRE(n == 0 || d_off, BATMAP_ERR_ARG, "d_offsets is NULL");
    std::lock_guard<std::mutex> lock(g_dense_mu);
    if (!g_dense) g_dense = new DenseWork();
    DenseWork &W = *g_dense;
    W.ev.create();
    W.ev.record(0, st);
    const uint64_t npairs = (uint64_t)n * (n > 0 ? n - 1 : 0) / 2;
    const BitsLayout L = bits_block_major(n, m);
    uint32_t *C = d_full;
    if (!C) {
        W.C.ensure(std::max<uint64_t>(npairs, 1));
        C = W.C.p;
    }
    W.state.ensure(4);
    W.total.ensure(1);
    W.bits.ensure(std::max<uint64_t>((uint64_t)L.kblocks * L.kb_stride, 32));
    BM_CUDA(cudaMemsetAsync(W.state.p, 0, 4 * sizeof(uint32_t), st));
    int *flags = reinterpret_cast<int *>(W.state.p + 2);
    enqueue_bits(d_off, d_tids, n, m, L, W.bits.p, flags, false, st);
    W.ev.record(1, st);
    std::vector<MmUnit> units;
    const bool add = contract_units(n, 0, L.kblocks, 0, 0.0, &units);
    const MmView view{W.bits.p, C, n, 0};
    if (!units.empty()) {
        if (add && npairs) BM_CUDA(cudaMemsetAsync(C, 0, npairs * sizeof(uint32_t), st));
        W.units.ensure(units.size());
        BM_CUDA(cudaMemcpyAsync(W.units.p, units.data(), units.size() * sizeof(MmUnit), cudaMemcpyHostToDevice, st));
        launch_contract(nullptr, view, W.units.p, (uint32_t)units.size(), W.state.p, st, nullptr,
                        g_dense_timeout_test.exchange(0));
    }
    W.ev.record(2, st);
    enqueue_threshold(C, n, s, d_pairs, cap, &W.blocksums, W.total.p, st);
    W.ev.record(3, st);
    int state[4] = {0, 0, 0, 0};
    uint64_t total = 0;
    BM_CUDA(cudaMemcpyAsync(state, W.state.p, sizeof(state), cudaMemcpyDeviceToHost, st));
    BM_CUDA(cudaMemcpyAsync(&total, W.total.p, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
    BM_CUDA(cudaStreamSynchronize(st));
    W.timing.build_ms = W.ev.ms(0, 1);
    W.timing.compare_ms = W.ev.ms(1, 2);
    W.timing.compact_ms = W.ev.ms(2, 3);
    W.timing.pairs_ms = W.ev.ms(0, 3);
    W.timing.place_ms = W.timing.finalize_ms = 0.f;
    if (tout) *tout = W.timing;
    BM_REQUIRE(state[2] == 0, BATMAP_ERR_ARG, "tids must be < m");
    BM_REQUIRE(state[1] == 0, BATMAP_ERR_TIMEOUT, "dense tensor-core kernel: a bounded pipeline wait timed out");
    check_total(total);
    *n_out = total;
    if (total > cap)
        throw Error{BATMAP_ERR_CAPACITY, "d_pairs too small: " + std::to_string(total) + " pairs qualify"};
}

}  // namespace bm

extern "C" void batmap_test_dense_timeout(uint32_t spin_limit) { bm::set_dense_timeout_test(spin_limit); }

extern "C" batmap_status pair_support_dense(uint32_t m, uint32_t n, const uint64_t *d_offsets, const uint32_t *d_tids,
                                            uint32_t s, uint32_t *d_pairs, uint64_t cap, uint64_t *n_out,
                                            uint32_t *d_full, batmap_timing *timing, cudaStream_t stream) {
    try {
        bm::run_dense(m, n, d_offsets, d_tids, s, d_pairs, cap, n_out, d_full, timing, stream);
        return BATMAP_OK;
    } catch (const bm::Error &e) {
        bm::set_error(e.msg);
        return e.code;
    } catch (...) {
        bm::set_error("unexpected internal error");
        return BATMAP_ERR_INTERNAL;
    }
}

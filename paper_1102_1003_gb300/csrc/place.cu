// Parallel cuckoo placement (Sec. II-A, generalised to d copies in d + 1
// tables) and the BatMap bytes (Sec. II, Sec. III-A), fused per item.
//
// Each thread carries one copy of one element.  Copy c starts in table c; a
// copy is swapped into its slot of table t; the evicted occupant (if any)
// continues in table t + 1 (cyclic).  Swapping a copy with another copy of the
// same element leaves the table unchanged and the element continues in the
// next table, so its copies always end in distinct tables.  Atomic exchanges
// conserve copies; a chain longer than max_moves drops the copy it holds.
// Afterwards every element with exactly d copies gets its d bytes; the others
// are failed insertions, counted per chunk and marked in a bit mask.
//
// Placement is random exchanges on a table of one 32-bit entry per slot, four
// times the BatMap's bytes.  Measured rates of random accesses by all SMs
// (G/s): exchanges 1,130 in shared memory, 129 in L2 (up to 32 MB), 40 at 256 MB
// and 28 at 2 GB; loads 272 in L2; byte stores 126 in L2.  So an item's table
// lives where those are cheap, from its first exchange to its last byte:
//   - up to 8,192 slots per table (k_place_small): in the shared memory of one
//     CTA, beside the item's slots in every table, computed once;
//   - above (k_place_large): in L2.  Items go in batches, alternately through
//     two regions of PLACE_L2_BYTES in all (or two sequences of batches, two
//     regions each); a launch inserts one batch and forms the bytes of the one
//     before, so that long chains do not hold the chip up.  Bytes are formed slot
//     by slot from a coalesced pass over the table:
//     one load in another table per copy tells which tables hold the element (no
//     byte is stored at random).  Entries carry an epoch above the tid, so a
//     region is not cleared between batches.
// Before, one launch placed all items through one table in DRAM and another looked
// every element up in it: at m = 2^22, 5%, n = 8,192 (51.5 GB of table) builds took
// 126 ms, and take 70.  At the rates above the exchanges, loads and writes of half
// those items come to 26 ms, and take 36.
#include <algorithm>
#include <type_traits>

#include "compare.cuh"
#include "place.cuh"
#include "scan.cuh"

namespace bm {
namespace place {

constexpr uint32_t SMALL_RLOG = 13;
constexpr uint32_t FIRST_MOVES = 16;  // of a chain before it waits for the others
static_assert(5u << SMALL_RLOG <= 1u << 16, "a slot of the widest table in 16 bits");
static_assert(SMALL_RLOG < PLACE_QUEUES, "a queue per width in shared memory");
constexpr uint64_t PLACE_L2_BYTES = 96ull << 20;
constexpr uint32_t SEQS = 2;
constexpr uint64_t SEQ_REGION = 22ull << 20;
static_assert(SEQS <= 1 + SideStream::MORE, "a stream for each");
constexpr int LTPB = 128;
constexpr uint32_t SUBS = LTPB / 32;                       // a warp per part of a CTA's task
constexpr uint32_t A_SUB = 256, A_ELEMS = SUBS * A_SUB;    // elements of a warp's, a CTA's insertions
constexpr uint32_t B_SUB = 512, B_SLOTS = SUBS * B_SUB;    // slots of a warp's, a CTA's bytes
constexpr uint32_t B_PASS = 512;                           // slots packed at a time, and the list's capacity
constexpr uint32_t A_ROUND = 128;                          // elements inserted at a time
static_assert(A_ROUND * 4 <= B_PASS, "the losers of a table's insertions fit behind what the list may hold");
constexpr size_t LARGE_SMEM = SUBS * (B_PASS * 8 + B_PASS);

// Byte layout: 2-of-3 has the indicator in bit 7 over a 7-bit code; d >= 3 the
// missing table in the top bits over a 6-bit (d = 3) or 5-bit (d = 4) code.
template <int NT>
__device__ __forceinline__ uint32_t byte_of(uint32_t has, uint32_t t, uint32_t code) {
    if constexpr (NT == 3) {  // 1 on the copy whose twin sits in the cyclic predecessor table (Fig. 3)
        return (((has >> ((t + 2) % 3)) & 1u) << 7) | code;
    } else {
        const uint32_t missing = __ffs(~has & ((1u << NT) - 1u)) - 1;
        return (missing << (NT == 4 ? 6 : 5)) | code;
    }
}

// Slot of position h = pi mod r in table t of NT interleaved in blocks of
// 2^shift; Slot is 32 bits wide where NT r fits.
template <int NT, typename Slot>
__device__ __forceinline__ Slot slot_of_h(uint32_t t, uint32_t h, uint32_t shift) {
    const uint32_t low = h & ((1u << shift) - 1u);
    return (Slot)NT * (h - low) + low + ((Slot)t << shift);
}
constexpr uint32_t SLOT32_RLOG = 28;

// Cycle walking with the round keys of a table.
__device__ __forceinline__ uint32_t pi_by(const PermView &P, const uint4 &k, uint32_t x) {
    uint32_t v = P.pass(k, x);
    while (v >= P.m) v = P.pass(k, v);
    return v;
}

// pi_t(x), the round keys of table t read by index from the kernel's parameters.
__device__ __forceinline__ uint32_t pi_of(const PermView &P, uint32_t t, uint32_t x) {
    if (P.table) return __ldg(&P.table[(uint64_t)t * P.m + x]);
    const uint4 k = P.key[t];
    return pi_by(P, k, x);
}

// Records the failures of 32 consecutive elements, the w-th of the item.
__device__ __forceinline__ void record(const PlaceJob &J, uint32_t item, uint32_t w, bool failed, uint32_t lane) {
    const uint32_t bits = __ballot_sync(0xffffffffu, failed);
    if (lane == 0) {
        const uint64_t chunk = J.chunk0[item] + w / (CHUNK / 32);
        J.mask[chunk * (CHUNK / 32) + w % (CHUNK / 32)] = bits;
        if (bits) atomicAdd((unsigned long long *)&J.fails[chunk], (unsigned long long)__popc(bits));
    }
}

// Has the check that runs beside the placement refused the input?  Equal tids (or a table
// that is no permutation) send all copies to a few slots, where every chain takes all its
// moves, one exchange after the other on one word: chains look every POLL moves, items and
// tasks before they begin.  A task's look may be answered by L1 (a launch old at most): the
// flags are one line for all SMs, and reading it in L2 for every task took k_place_large 6%
// (m = 2^22, 5%, n = 2,048: 17.75 -> 18.9 ms) to 40% (0.1%).
// Chains of the default max_loop, of 96 to 160 moves, do not look (every 64 moves: quadruples
// of n = 1,000, m = 100,000 2.36 -> 2.39 ms).
constexpr uint32_t POLL = 256;
__device__ __forceinline__ bool refused(const PlaceJob &J) {
    if (!J.refused) return false;
    const volatile int *f = J.refused;
    return (f[0] | f[1] | f[2] | f[3]) != 0;
}

// One CTA per item, items from a queue.  Dynamic shared memory: NT 2^rlog
// entries (first the tids, then element indices, then the item's bytes); per
// element and table its slot (16 bits: at most 5 * 8,192 slots) and code (8 bits, 0:
// not a tid); per element the tables that hold it (8 bits).  Each pi_t(x) is
// computed once: chains and bytes read slots and codes.
template <int NT>
__global__ void __launch_bounds__(1024) k_place_small(const __grid_constant__ PlaceJob J,
                                                      const __grid_constant__ PermView P, uint32_t cap) {
    extern __shared__ __align__(16) uint32_t table[];
    __shared__ uint32_t s_item, s_late;
    const uint32_t slots = (uint32_t)NT << J.rlog, rm = (1u << J.rlog) - 1u;
    uint8_t *bytes = reinterpret_cast<uint8_t *>(table);
    uint16_t *slot = reinterpret_cast<uint16_t *>(table + slots);  // [cap][NT]
    uint8_t *code = reinterpret_cast<uint8_t *>(slot + NT * cap);  // [cap][NT]
    uint8_t *held = code + NT * cap;                               // [cap]
    uint32_t *late = reinterpret_cast<uint32_t *>(held);           // [cap / 4], before held is written
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, tpb = blockDim.x, warps = tpb / 32;
    uint4 *t4 = reinterpret_cast<uint4 *>(table);
    for (;;) {
        if (threadIdx.x == 0) {
            const uint32_t next = atomicAdd(J.queue, 1u);
            s_item = refused(J) ? J.count : next;
            s_late = 0;
        }
        __syncthreads();
        if (s_item >= J.count) break;
        const uint32_t item = J.items[s_item];
        const uint64_t e0 = J.off[item];
        const uint32_t size = (uint32_t)(J.off[item + 1] - e0);  // <= cap, <= slots
        for (uint32_t e = threadIdx.x; e < size; e += tpb) table[e] = J.tids[e0 + e];
        __syncthreads();
        if (P.table) {
            for (uint32_t e = threadIdx.x; e < size; e += tpb) {
                const uint32_t x = table[e];
                uint32_t v[NT];
#pragma unroll
                for (uint32_t t = 0; t < NT; t++) v[t] = x < P.m ? __ldg(&P.table[(uint64_t)t * P.m + x]) : 0;
#pragma unroll
                for (uint32_t t = 0; t < NT; t++) {
                    slot[e * NT + t] = (uint16_t)slot_of_h<NT, uint32_t>(t, v[t] & rm, J.shift);
                    code[e * NT + t] = x < P.m ? (uint8_t)((v[t] >> J.shift) + 1u) : 0;  // else rejected by validation
                }
            }
        } else {
            // pi_t(x): cycle walking takes 1 to 4 passes on average, the longest of 32 lanes far more, so
            // a lane that is done takes the warp's next (element, table)
            const uint32_t total = NT * size;
            uint32_t taken = 0, idx = 0, v = 0;
            bool busy = false;
            for (;;) {
                const uint32_t idle = __ballot_sync(0xffffffffu, !busy);
                if (!busy) {
                    const uint32_t k = taken + __popc(idle & ((1u << lane) - 1u));
                    idx = ((k >> 5) * warps + warp) * 32u + (k & 31u);
                    if (idx < total) {
                        v = table[idx / NT];
                        busy = v < P.m;  // else rejected by validation
                        if (!busy) code[idx] = 0, slot[idx] = 0;
                    }
                }
                taken += __popc(idle);
                if (__any_sync(0xffffffffu, busy)) {
                    if (busy) {
                        v = P.pass(P.key[idx % NT], v);
                        if (v < P.m) {
                            slot[idx] = (uint16_t)slot_of_h<NT, uint32_t>(idx % NT, v & rm, J.shift);
                            code[idx] = (uint8_t)((v >> J.shift) + 1u);
                            busy = false;
                        }
                    }
                } else if (((taken >> 5) * warps + warp) * 32u >= total) {
                    break;
                }
            }
        }
        __syncthreads();
        for (uint32_t k = threadIdx.x; k < slots / 4; k += tpb) t4[k] = make_uint4(EMPTY, EMPTY, EMPTY, EMPTY);
        for (uint32_t k = slots / 4 * 4 + threadIdx.x; k < slots; k += tpb) table[k] = EMPTY;
        __syncthreads();
        // the chain of copy (e, t) goes on; true: it ended in an empty slot
        auto walk = [&](uint32_t &e, uint32_t &t, uint32_t moves) {
            for (uint32_t mv = 0; mv < moves; mv++) {
                e = atomicExch(&table[slot[e * NT + t]], e);
                if (e == EMPTY) return true;
                t = t + 1 == NT ? 0 : t + 1;  // the same element: another of its copies, go on
            }
            return false;
        };
        // Few chains are long, and those of elements that cannot be placed take all their moves: they wait
        // in a list until the rest is in, then go side by side and not one after another (3-of-4 and 4-of-5
        // sets of n = 1,000, m = 100,000: launches of 120 us each, passes 1833 -> 1553 and 2631 -> 2412 us
        // with the next rule for those in L2).
        const uint32_t soon = min(J.max_moves, FIRST_MOVES), rest = J.max_moves - soon;
        auto finish = [&](uint32_t e, uint32_t t) {
            for (uint32_t left = rest;;) {
                const uint32_t moves = min(left, POLL);
                if (walk(e, t, moves) || !(left -= moves) || refused(J)) return;
            }
        };
        for (uint32_t c = 0; c < NT - 1; c++)
            for (uint32_t k = threadIdx.x; k < size; k += tpb) {
                if (!code[k * NT]) continue;
                uint32_t e = k, t = c;
                if (walk(e, t, soon) || !rest) continue;
                const uint32_t at = atomicAdd(&s_late, 1u);
                if (at < cap / 4) late[at] = e | t << 16;
                else finish(e, t);
            }
        __syncthreads();
        for (uint32_t k = threadIdx.x; k < min(s_late, cap / 4); k += tpb) {
            finish(late[k] & 0xFFFFu, late[k] >> 16);
        }
        __syncthreads();
        for (uint32_t e = threadIdx.x; e < (size + 31u) / 32u * 32u; e += tpb) {
            bool failed = false;
            if (e < size) {
                uint32_t has = 0;
#pragma unroll
                for (uint32_t t = 0; t < NT; t++)
                    has |= (table[slot[e * NT + t]] == e ? 1u : 0u) << t;
                const bool valid = code[e * NT] != 0, whole = valid && __popc(has) == NT - 1;
                failed = valid && !whole;
                held[e] = whole ? (uint8_t)has : 0;
            }
            record(J, item, e / 32, failed, lane);
        }
        __syncthreads();
        for (uint32_t k = threadIdx.x; k < slots / 16; k += tpb) t4[k] = make_uint4(0, 0, 0, 0);
        for (uint32_t k = slots / 16 * 4 + threadIdx.x; 4 * k < slots; k += tpb) table[k] = 0;
        __syncthreads();
        for (uint32_t e = threadIdx.x; e < size; e += tpb) {
            const uint32_t has = held[e];
#pragma unroll
            for (uint32_t t = 0; t < NT; t++)
                if ((has >> t) & 1u)
                    bytes[slot[e * NT + t]] = (uint8_t)byte_of<NT>(has, t, code[e * NT + t]);
        }
        __syncthreads();
        uint8_t *to = J.out + J.base[item];
        if (((slots | J.base[item]) & 15u) == 0) {
            uint4 *out = reinterpret_cast<uint4 *>(to);
            for (uint32_t k = threadIdx.x; k < slots / 16; k += tpb) out[k] = t4[k];
        } else {  // BatMaps of less than 48 bytes, and those behind them
            for (uint32_t k = threadIdx.x; k < slots; k += tpb) to[k] = bytes[k];
        }
        __syncthreads();
    }
}

// ---- items whose tables live in L2 ----------------------------------------------

struct LargeItem {
    uint64_t table;       // first word of its table in the scratch
    uint32_t item, rlog, epoch;
    uint32_t first_a, first_b, na, nb;  // its CTAs' tasks: insertions, bytes
    uint32_t pad;
};
// A displaced copy's next table and the moves of its chain so far (at most MAX_MOVES).
__host__ __device__ constexpr uint32_t chain_word(uint32_t t, uint32_t moves) { return t | moves << 3; }
__host__ __device__ constexpr uint32_t chain_table(uint32_t w) { return w & 7u; }
__host__ __device__ constexpr uint32_t chain_moves(uint32_t w) { return w >> 3; }
static_assert(chain_moves(chain_word(4, MAX_MOVES - 1)) + 1 == MAX_MOVES && chain_table(chain_word(4, MAX_MOVES - 1)) == 4,
              "a chain's count reaches its limit");

struct LargeTask {
    uint32_t q, k;  // k-th insertion task, or (LARGE_BYTES set) byte task, of large item q
};
constexpr uint32_t LARGE_BYTES = 1u << 31;

__global__ void k_large_tasks(const LargeItem *items, LargeTask *tasks) {
    const LargeItem I = items[blockIdx.x];
    for (uint32_t k = threadIdx.x; k < I.na; k += blockDim.x) tasks[I.first_a + k] = {blockIdx.x, k};
    for (uint32_t k = threadIdx.x; k < I.nb; k += blockDim.x) tasks[I.first_b + k] = {blockIdx.x, k | LARGE_BYTES};
}

// One CTA per task, a warp per part of it: a batch's insertions, then the
// bytes of the batch before (inserted by the launch before, in the other
// region).  drops[q]: copies that item q lost.
// Slot of 32 bits where all slots fit and every BatMap starts at a multiple of 4 bytes (a test of
// that at the stores took 0.35%), else of 64.
template <int NT, typename Slot>
__global__ void __launch_bounds__(LTPB, 8)
k_place_large(const __grid_constant__ PlaceJob J, const __grid_constant__ PermView P, const LargeItem *__restrict__ items,
              const LargeTask *__restrict__ tasks, uint32_t tbits, uint32_t hbits, bool known, uint32_t *scratch,
              uint32_t *drops) {
    extern __shared__ __align__(16) uint2 s_large[];       // per warp: the list, then the bytes
    uint2 *list = s_large + (threadIdx.x >> 5) * (B_PASS + B_PASS / 8);  // a pass's entries: entry, slot
    uint8_t *bytes = reinterpret_cast<uint8_t *>(list + B_PASS);
    uint32_t *words = reinterpret_cast<uint32_t *>(bytes);
    const uint32_t tidmask = (1u << tbits) - 1u, lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
    // an entry: epoch | the bits of pi_t(x) from r on, hbits of them | tid (known: position and entry
    // together give pi_t(x); else it is computed again)
    const uint32_t eshift = tbits + hbits, same = ~(((1u << hbits) - 1u) << tbits);
    const LargeTask task = tasks[blockIdx.x];
    const struct { uint32_t q, k; bool bytes; } T{task.q, task.k & ~LARGE_BYTES, (task.k & LARGE_BYTES) != 0};
    const LargeItem I = items[T.q];
    const uint32_t sub = threadIdx.x >> 5;
    uint32_t *table = scratch + I.table;
    const uint32_t rlog = I.rlog, rm = (1u << rlog) - 1u, tag = I.epoch << eshift;
    const uint64_t e0 = J.off[I.item], size = J.off[I.item + 1] - e0;
    const uint32_t *tids = J.tids + e0;
    if (J.refused) {
        const int4 f = __ldca(reinterpret_cast<const int4 *>(J.refused));
        if (__any_sync(0xffffffffu, f.x | f.y | f.z | f.w)) return;
    }
    if (!T.bytes) {
        // First every copy's own exchange, all lanes in one table, four in flight; the displaced copies
        // go to a list, whose chains run on with full warps while it is long enough.
        const uint64_t b0 = (uint64_t)T.k * A_ELEMS + sub * A_SUB, b1 = min(size, b0 + A_SUB);
        uint32_t waiting = 0;  // entries of the list: tid, chain_word
        const uint32_t soon = min(J.max_moves, POLL);
        auto chains = [&](uint32_t least) {
            while (waiting >= least) {
                const uint32_t n = min(waiting, 32u);
                waiting -= n;
                const uint2 c = lane < n ? list[waiting + lane] : make_uint2(0, 0);
                uint2 next = make_uint2(0, 0);
                bool lost = false;
                if (lane < n) {
                    const uint32_t t = chain_table(c.y), pi = pi_of(P, t, c.x), high = known ? (pi >> rlog) << tbits : 0;
                    const uint32_t old = atomicExch(&table[slot_of_h<NT, Slot>(t, pi & rm, J.shift)], tag | high | c.x);
                    const uint32_t moves = chain_moves(c.y) + 1;
                    lost = (old >> eshift) == I.epoch;
                    next = make_uint2(old & tidmask, chain_word(t + 1 == NT ? 0 : t + 1, moves));
                    if (lost && moves >= soon && (moves >= J.max_moves || (moves % POLL == 0 && refused(J)))) {
                        atomicAdd(&drops[T.q], 1u);
                        lost = false;
                    }
                }
                const uint32_t mask = __ballot_sync(0xffffffffu, lost);
                __syncwarp();
                if (lost) list[waiting + __popc(mask & below)] = next;
                waiting += __popc(mask);
                __syncwarp();
            }
        };
        for (uint64_t b = b0; b < b1; b += A_ROUND) {
            uint32_t x[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const uint64_t e = b + 32u * i + lane;
                x[i] = e < b1 ? __ldcs(&tids[e]) : 0xFFFFFFFFu;  // tids >= m: rejected by validation
            }
#pragma unroll
            for (uint32_t c = 0; c < NT - 1; c++) {
                uint32_t old[4];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    old[i] = 0;
                    if (x[i] < P.m) {
                        const uint32_t pi = pi_of(P, c, x[i]), high = known ? (pi >> rlog) << tbits : 0;
                        old[i] = atomicExch(&table[slot_of_h<NT, Slot>(c, pi & rm, J.shift)], tag | high | x[i]);
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const bool lost = (old[i] >> eshift) == I.epoch;  // (epochs start at 1)
                    const uint32_t mask = __ballot_sync(0xffffffffu, lost);
                    if (lost) list[waiting + __popc(mask & below)] = make_uint2(old[i] & tidmask, chain_word(c + 1, 1));
                    waiting += __popc(mask);
                }
                __syncwarp();
                // room for the next table's losers, and full warps
                if (waiting > B_PASS - A_ROUND) chains(B_PASS - A_ROUND);
            }
            chains(32);
        }
        chains(1);
    } else {
        // L1 may hold lines of an earlier use of the region: loads go to L2
        const bool lossy = drops[T.q] != 0;
        const uint64_t slots = (uint64_t)NT << rlog, s0 = (uint64_t)T.k * B_SLOTS + sub * B_SUB;
        const uint32_t low = (1u << J.shift) - 1u;
        uint8_t *out = J.out + J.base[I.item];
        const bool aligned = sizeof(Slot) == 4 || ((slots | J.base[I.item]) & 3u) == 0;
        // The entries of a pass: each looks into the next table.  `same`: all lie in one table, t0,
        // at positions h0 on; its next one's keys are read once and no slot is taken apart.
        auto entries = [&](auto one, Slot s, uint32_t used) {
            constexpr bool ONE = decltype(one)::value;
            const Slot seg0 = s >> J.shift;
            const uint32_t t0 = ONE ? (uint32_t)(seg0 % NT) : 0, h0 = ONE ? ((uint32_t)(seg0 / NT) << J.shift) | ((uint32_t)s & low) : 0;
            const uint32_t next0 = t0 + 1 == NT ? 0 : t0 + 1;
            const uint4 key = P.key[next0];
            const uint32_t *row = P.table + (uint64_t)next0 * P.m;
            for (uint32_t k0 = 0; k0 < used; k0 += 64) {
                // two entries a lane: their looks together
                uint2 c[2];
                uint32_t t[2], h[2], y[2];
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    const uint32_t k = k0 + 32u * u + lane;
                    y[u] = 0;
                    if (k >= used) continue;
                    c[u] = list[k];
                    t[u] = t0;
                    h[u] = h0 + c[u].y;
                    uint32_t next = next0, pi;
                    const uint32_t x = c[u].x & tidmask;
                    if (!ONE) {
                        const Slot at = s + c[u].y, seg = at >> J.shift;
                        t[u] = (uint32_t)(seg % NT);
                        h[u] = ((uint32_t)(seg / NT) << J.shift) | ((uint32_t)at & low);
                        next = t[u] + 1 == NT ? 0 : t[u] + 1;
                        pi = pi_of(P, next, x);
                    } else {
                        pi = P.table ? __ldg(&row[x]) : pi_by(P, key, x);
                    }
                    y[u] = __ldcg(&table[slot_of_h<NT, Slot>(next, pi & rm, J.shift)]);
                }
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    if (k0 + 32u * u + lane >= used) continue;
                    const uint32_t w = c[u].x, x = w & tidmask;
                    const bool here = ((y[u] ^ w) & same) == 0;
                    uint32_t has;
                    bool whole = true;
                    if (NT == 3 && !lossy) {  // in the next table or the one after
                        const uint32_t at = t[u] + (here ? 1 : 2);
                        has = 1u << t[u] | 1u << (at >= NT ? at - NT : at);
                    } else {
                        // the tables that hold x: t and, of the others, all but one; without lost copies the
                        // last need not be looked at
                        uint32_t at = t[u] + 1 == NT ? 0 : t[u] + 1, found = here ? 2 : 1;
                        has = 1u << t[u] | (here ? 1u << at : 0u);
                        for (uint32_t o = 2; o < NT; o++) {
                            at = at + 1 == NT ? 0 : at + 1;
                            if (!lossy && (found < o || o + 1 == NT)) {  // the missing table is known, or left to the last
                                if (found == NT - 1) break;
                                has |= 1u << at;
                                found++;
                            } else if (((__ldcg(&table[slot_of_h<NT, Slot>(at, pi_of(P, at, x) & rm, J.shift)]) ^ w) & same) == 0) {
                                has |= 1u << at;
                                found++;
                            }
                        }
                        whole = found == NT - 1;
                    }
                    if (whole) {
                        const uint32_t pi = known ? (((w >> tbits) & ((1u << hbits) - 1u)) << rlog) | h[u] : pi_of(P, t[u], x);
                        bytes[c[u].y] = (uint8_t)byte_of<NT>(has, t[u], (pi >> J.shift) + 1u);
                    }
                }
            }
        };
        for (uint64_t s = s0; s < min(slots, s0 + B_SUB); s += B_PASS) {
            // the used slots of the pass, packed: few of a table's slots are used, and each costs a
            // permutation and a load
            uint32_t used = 0;
#pragma unroll
            for (uint32_t i = 0; i < B_PASS / 128; i++) {
                const uint32_t o = 128u * i + 4u * lane;
                const uint4 v = s + o < slots ? __ldcg(reinterpret_cast<const uint4 *>(table + s + o)) : make_uint4(0, 0, 0, 0);
                const uint32_t w[4] = {v.x, v.y, v.z, v.w};
                words[o / 4] = 0;
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const bool hit = (w[j] >> eshift) == I.epoch;
                    const uint32_t mask = __ballot_sync(0xffffffffu, hit);
                    if (hit) list[used + __popc(mask & below)] = make_uint2(w[j], o + j);
                    used += __popc(mask);
                }
            }
            __syncwarp();
            if (1u << J.shift >= B_PASS) entries(std::true_type{}, (Slot)s, used);  // (passes and tables' blocks are powers of two)
            else entries(std::false_type{}, (Slot)s, used);
            __syncwarp();
#pragma unroll
            for (uint32_t i = 0; i < B_PASS / 128; i++) {
                const uint32_t o = 128u * i + 4u * lane;
                if (aligned) {
                    if (s + o < slots) __stcs(reinterpret_cast<uint32_t *>(out + s + o), words[o / 4]);
                } else {
                    for (uint32_t j = o; j < o + 4 && s + j < slots; j++) out[s + j] = bytes[j];
                }
            }
            __syncwarp();
        }
        if (lossy) {  // this task's share of the elements: which ones failed
            const uint64_t words = (size + 31) / 32, parts = (uint64_t)I.nb * SUBS, part = (uint64_t)T.k * SUBS + sub;
            for (uint64_t w = words * part / parts; w < words * (part + 1) / parts; w++) {
                const uint64_t e = 32 * w + lane;
                bool failed = false;
                if (e < size) {
                    const uint32_t x = tids[e];
                    if (x < P.m) {
                        uint32_t found = 0;
                        for (uint32_t t = 0; t < NT; t++)
                            found += ((__ldcg(&table[slot_of_h<NT, Slot>(t, pi_of(P, t, x) & rm, J.shift)]) ^ (tag | x)) & same) == 0;
                        failed = found != NT - 1;
                    }
                }
                record(J, I.item, (uint32_t)w, failed, lane);
            }
        }
    }
}

// Words of an item's table in a region: whole 16-byte loads, also where the range is small.
template <int NT>
static uint64_t table_words(uint32_t rlog) {
    return (((uint64_t)NT << rlog) + 63) / 64 * 64;
}

// The large items in order of the list (widest first): batches, places and tasks.
template <int NT>
static void place_large(const PlaceJob &job, const PermView &P, const std::vector<PlaceItem> &list, uint32_t least_rlog,
                        SideStream &streams, bool may_widen = true) {
    cudaStream_t st = streams.main();
    uint32_t tbits = 1;
    while (tbits < 30 && (1ull << tbits) < P.m) tbits++;
    // the bits of pi_t(x) that its position does not give go along in the entry where there is room
    // for them beside at least four bits of epoch
    uint32_t hbits = tbits > list.back().rlog ? tbits - list.back().rlog : 0;
    const bool known = tbits + hbits <= 28;
    if (!known) hbits = 0;
    const uint32_t epochs = (1u << (32 - tbits - hbits)) - 1u;
    const uint64_t widest = table_words<NT>(list[0].rlog);
    uint64_t total = 0;
    for (const PlaceItem &I : list) total += table_words<NT>(I.rlog);
    // Two sequences of launches where there are batches for both and room for their regions: the end of
    // one's launch, a few long chains of exchanges, runs beside the body of the other's.  m = 2^22, 5%,
    // n = 2,048 (6.3 MB an item): one sequence 21.0 ms, two with 4 items a region 19.4, with 3 items
    // 17.9 (75 MB in use), three with 2 items 17.9; zipf m = 1 M, n = 2,000 (up to 25 MB) 2.2 and 2.0 ms.
    // With four and five tables the copies fill more of their slots and the chains are longer, so a
    // region takes 16 of the widest items, up to twice as much, where two sequences of such batches
    // come of it (a launch of two or four items ends with one's chains).  m = 10^6, 5%, n = 500, d = 4:
    // 9.4 -> 7.4 ms; m = 16 M, 1%, n = 100, from a caller's permutation table 12.2 -> 10.1.  Not for
    // more than 16: m = 120,000, 20%, n = 2,000 (1 MB an item): 5.9 -> 6.2 in twice as much.
    const uint64_t wide = std::min(16 * 4 * widest, 2 * SEQ_REGION);
    const uint64_t reg = may_widen && NT > 3 && wide > SEQ_REGION && 4 * total >= 2 * SEQS * wide ? wide : SEQ_REGION;
    const uint64_t most = (PLACE_L2_BYTES + 2 * SEQS * (reg - SEQ_REGION)) / 4;  // words of all
    const uint64_t part = std::max<uint64_t>(widest, reg / 4);
    // Everything in one batch where it fits: insertions, then bytes (two batches of the above triples' sets
    // took three launches, each as long as its longest chains).
    const bool once = total <= PLACE_L2_BYTES / 4;
    const uint32_t seqs = !once && 2 * SEQS * part <= most && total >= 2 * SEQS * part ? SEQS : 1;
    const uint64_t region = once ? total : (seqs > 1 ? part : std::max<uint64_t>(widest, most / 2)) / 64 * 64;  // (16-byte loads)
    static const bool ready = [] {
        BM_CUDA(cudaFuncSetAttribute(k_place_large<NT, uint32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LARGE_SMEM));
        BM_CUDA(cudaFuncSetAttribute(k_place_large<NT, uint64_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LARGE_SMEM));
        return true;
    }();
    (void)ready;
    std::vector<LargeItem> items(list.size());
    std::vector<size_t> first;  // first item of each batch
    uint64_t fill = 0;
    for (size_t q = 0; q < list.size(); q++) {
        const uint64_t words = table_words<NT>(list[q].rlog);
        if (first.empty() || fill + words > region) {
            first.push_back(q);
            fill = 0;
        }
        const uint32_t b = (uint32_t)first.size() - 1;
        LargeItem &I = items[q];
        I.table = b % (2 * seqs) * region + fill;
        I.item = list[q].item;
        I.rlog = list[q].rlog;
        I.epoch = 1 + b / (2 * seqs) % epochs;
        I.na = (uint32_t)((list[q].size + A_ELEMS - 1) / A_ELEMS);
        I.nb = (uint32_t)((words + B_SLOTS - 1) / B_SLOTS);
        fill += words;
    }
    const uint32_t nb = (uint32_t)first.size();
    first.push_back(list.size());
    std::vector<uint64_t> start;  // first task of each launch: the insertions of batch b, the bytes of the one before in its sequence
    uint64_t pos = 0;
    for (uint32_t b = 0; b < nb + seqs; b++) {
        start.push_back(pos);
        if (b < nb)
            for (size_t q = first[b]; q < first[b + 1]; q++) {
                items[q].first_a = (uint32_t)pos;
                pos += items[q].na;
            }
        if (b >= seqs && b - seqs < nb)
            for (size_t q = first[b - seqs]; q < first[b - seqs + 1]; q++) {
                items[q].first_b = (uint32_t)pos;
                pos += items[q].nb;
            }
    }
    start.push_back(pos);
    BM_REQUIRE(pos < (1ull << 31), BATMAP_ERR_ARG, "too many placement tasks");
    // scratch words: drops (zeroed) | items | tasks | the regions
    auto up = [](uint64_t w) { return (w + 63) / 64 * 64; };
    const uint64_t o_items = up(items.size()), o_tasks = o_items + up(items.size() * sizeof(LargeItem) / 4),
                   o_reg = o_tasks + up(pos * sizeof(LargeTask) / 4), regions = std::min<uint64_t>(nb, 2 * seqs);
    uint32_t *w;
    try {
        w = scratch_table(o_reg + regions * region).p;
    } catch (const Error &e) {
        if (e.code != BATMAP_ERR_NOMEM || reg == SEQ_REGION) throw;
        return place_large<NT>(job, P, list, least_rlog, streams, false);  // no room for the larger regions
    }
    BM_CUDA(cudaMemsetAsync(w, 0, o_items * 4, st));
    BM_CUDA(cudaMemcpyAsync(w + o_items, items.data(), items.size() * sizeof(LargeItem), cudaMemcpyHostToDevice, st));
    const LargeItem *d_items = reinterpret_cast<const LargeItem *>(w + o_items);
    LargeTask *d_tasks = reinterpret_cast<LargeTask *>(w + o_tasks);
    k_large_tasks<<<(unsigned)items.size(), 128, 0, st>>>(d_items, d_tasks);
    BM_CHECK_LAUNCH();
    cudaStream_t seq[SEQS] = {st};
    for (uint32_t c = 1; c < seqs; c++) seq[c] = streams.more(c - 1);
    for (uint32_t b = 0; b < nb + seqs; b++) {
        st = seq[b % seqs];
        // a region's first use, or all epochs used: clear it
        if (b < nb && b / (2 * seqs) % epochs == 0)
            BM_CUDA(cudaMemsetAsync(w + o_reg + b % (2 * seqs) * region, 0, region * 4, st));
        const unsigned grid = (unsigned)(start[b + 1] - start[b]);
        if (!grid) continue;
        if (list[0].rlog <= SLOT32_RLOG && least_rlog >= 2)
            k_place_large<NT, uint32_t><<<grid, LTPB, LARGE_SMEM, st>>>(job, P, d_items, d_tasks + start[b], tbits, hbits,
                                                                        known, w + o_reg, w);
        else
            k_place_large<NT, uint64_t><<<grid, LTPB, LARGE_SMEM, st>>>(job, P, d_items, d_tasks + start[b], tbits, hbits,
                                                                        known, w + o_reg, w);
        BM_CHECK_LAUNCH();
    }
}

template <int NT>
static void place_all(const PlaceJob &job, const PermView &P, std::vector<PlaceItem> &list, uint32_t *d_list,
                      SideStream &streams) {
    cudaStream_t side = streams.side();
    static const bool ready = [] {
        BM_CUDA(cudaFuncSetAttribute(k_place_small<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024 - 1024));
        return true;
    }();
    (void)ready;
    auto smem_of = [](uint32_t rlog, uint64_t cap) { return ((uint64_t)NT << rlog) * 4 + cap * (3 * NT + 1); };
    auto cap_of = [](uint64_t size) { return std::max<uint64_t>(32, (size + 31) / 32 * 32); };
    // items for L2, widest first, then those for shared memory, runs of equal width
    std::stable_sort(list.begin(), list.end(), [](const PlaceItem &a, const PlaceItem &b) { return a.rlog > b.rlog; });
    const uint32_t least = list.back().rlog;  // of all: BatMaps lie one behind the other
    const auto mid = std::stable_partition(list.begin(), list.end(), [&](const PlaceItem &I) {
        // (the tids are staged where the table will be: no more of them than slots)
        return I.rlog > SMALL_RLOG || I.size > ((uint64_t)NT << I.rlog) || smem_of(I.rlog, cap_of(I.size)) > 225 * 1024;
    });
    std::vector<uint32_t> ids;
    for (const PlaceItem &I : list) ids.push_back(I.item);
    BM_CUDA(cudaMemcpyAsync(d_list, ids.data(), ids.size() * 4, cudaMemcpyHostToDevice, side));
    // (widths side by side on streams of their own: triples 2% slower, quadruples 10%)
    uint32_t launch = 0;
    if (mid != list.begin()) place_large<NT>(job, P, std::vector<PlaceItem>(list.begin(), mid), least, streams);
    for (size_t k = mid - list.begin(); k < list.size();) {
        size_t e = k;
        uint64_t most = 0;
        while (e < list.size() && list[e].rlog == list[k].rlog) most = std::max(most, list[e++].size);
        PlaceJob J = job;
        J.items = d_list + k;
        J.count = (uint32_t)(e - k);
        J.rlog = list[k].rlog;
        J.queue = job.queue + launch++;
        const uint32_t cap = (uint32_t)cap_of(most), smem = (uint32_t)smem_of(J.rlog, cap);
        // four elements a thread where the items fill their range; fewer where the items alone do not fill
        // the chip, and the time is that of one of them (n = 200, m = 10,000:
        // the pass 266 -> 253 us)
        uint32_t tpb = std::min(1024u, std::max(128u, (1u << J.rlog) / 8u));
        while (tpb < 512 && (uint64_t)J.count * tpb < (uint64_t)device_sms() * 1024) tpb *= 2;
        const uint32_t fit = std::max(1u, std::min(2048u / tpb, 226u * 1024u / (smem + 1024u)));
        k_place_small<NT><<<std::min(J.count, (uint32_t)device_sms() * fit), tpb, smem, side>>>(J, P, cap);
        BM_CHECK_LAUNCH();
        k = e;
    }
}

}  // namespace place

__global__ void k_perm_table(const __grid_constant__ PermView P, uint32_t tables, uint32_t *__restrict__ out) {
    const uint64_t total = (uint64_t)tables * P.m;
    for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < total; k += (uint64_t)gridDim.x * blockDim.x)
        out[k] = place::pi_of(P, (uint32_t)(k / P.m), (uint32_t)(k % P.m));
}

// A pass of the network is about 50 instructions.  Where 2^b is near m a warp takes one or
// two of them, 450 to 800 G/s; at 2^b = 2.6 m its slowest lane takes eight or nine, 100 G/s,
// against 272 G/s loads in L2.  So from 2^b = 1.5 m on, where the table stays small beside
// the batches in L2 and is read far more often than it is long.  n = 8,000, m = 25,000
// (2^16): 1474 -> 1200 us with the supports; triples and quadruples of n = 1,000,
// m = 100,000 (2^18): 2168 -> 1824 and 3367 -> 2683 us.
PermView place_perms(const PermView &P, uint32_t tables, uint64_t total, Workspace &ws, cudaStream_t st) {
    if (P.table || 2 * (1ull << (2 * P.half)) < 3ull * P.m || 4ull * tables * P.m > (16u << 20) || total < 16ull * P.m) return P;
    PermView T = P;
    WsBuf<uint32_t> table(ws, (uint64_t)tables * P.m);
    k_perm_table<<<(unsigned)std::min<uint64_t>(((uint64_t)tables * P.m + 255) / 256, 4096), 256, 0, st>>>(P, tables, table.p);
    BM_CHECK_LAUNCH();
    T.table = table.p;
    return T;
}

void enqueue_place(uint32_t tables, PlaceJob job, const PermView &P, std::vector<PlaceItem> list,
                   uint32_t *d_list, SideStream &streams) {
    if (list.empty()) return;
    job.max_moves = std::min(job.max_moves, MAX_MOVES);
    BM_CUDA(cudaMemsetAsync(job.queue, 0, PLACE_QUEUES * sizeof(uint32_t), streams.side()));
    if (tables == 3) place::place_all<3>(job, P, list, d_list, streams);
    if (tables == 4) place::place_all<4>(job, P, list, d_list, streams);
    if (tables == 5) place::place_all<5>(job, P, list, d_list, streams);
}

__global__ void k_failures(ItemView v, const uint32_t *mask, const uint64_t *offsets, uint32_t *f_item, uint32_t *f_tid) {
    uint64_t running = offsets[blockIdx.x];
    if (offsets[blockIdx.x + 1] == running) return;  // no failure in this chunk
    uint32_t item;
    uint64_t e0, e1;
    chunk_range(v, blockIdx.x, &item, &e0, &e1);
    for (int j = 0; j < PER_THREAD; j++) {
        const uint32_t k = (uint32_t)j * TPB + threadIdx.x;
        const bool fail = e0 + k < e1 && (mask[(uint64_t)blockIdx.x * (CHUNK / 32) + k / 32] >> (k & 31u)) & 1u;
        uint64_t tot;
        const uint64_t rank = block_exclusive_scan(fail ? 1 : 0, &tot);
        if (fail) {
            f_item[running + rank] = item;
            f_tid[running + rank] = v.tids[e0 + k];
        }
        running += tot;
    }
}

}  // namespace bm

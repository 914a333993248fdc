// Placement of the elements of all items and the bytes of their BatMaps, for
// 2-of-3, 3-of-4 and 4-of-5 sets.
#pragma once

#include "items.cuh"

namespace bm {

struct PlaceJob {
    const uint64_t *off;     // CSR
    const uint32_t *tids;
    const uint64_t *base;    // [n] first byte of item i in `out`
    const uint32_t *chunk0;  // [n] first chunk (CHUNK elements) of item i
    const uint32_t *items;   // a launch's items, all of range 2^rlog (set by the launches)
    uint32_t count, rlog, shift, max_moves;
    uint8_t *out;            // BatMap bytes (every byte of the items is written)
    uint64_t *fails;         // [chunks] zeroed; failed insertions per chunk
    uint32_t *mask;          // [chunks * CHUNK / 32] bit e: element e of the chunk failed
    uint32_t *queue;         // PLACE_QUEUES words
    const int *refused;      // 4 flags that the check of the lists and permutations beside the placement may set
                             // (BuildStat::err), or nullptr: the call is refused, and what is left to place is not placed
};

// Places all items of the list (ids, any order; d_list: room for as many ids on
// the device); tables: d + 1 (3, 4 or 5).  The wide ones go on the caller's stream and
// another, the rest on the side stream; the caller joins them.
struct PlaceItem {
    uint32_t item, rlog;
    uint64_t size;
};
constexpr uint32_t PLACE_QUEUES = 64;
// Moves of a chain, whatever the job asks for: 5 tables times the largest max_loop of a build
// are less; a pool's max_loop has no other bound (a move takes about a microsecond in L2).
constexpr uint32_t MAX_MOVES = 1u << 23;
void enqueue_place(uint32_t tables, PlaceJob job, const PermView &P, std::vector<PlaceItem> list,
                   uint32_t *d_list, SideStream &streams);

// The permutations that the placement of `total` elements reads: a table in ws, written on
// st, where computing them by cycle walking costs more, else P.
PermView place_perms(const PermView &P, uint32_t tables, uint64_t total, Workspace &ws, cudaStream_t st);

// F_i of every chunk with failures, in (item, tid) order: offsets[b] = first
// entry of chunk b (exclusive scan of the counts, with the total behind it).
__global__ void k_failures(ItemView v, const uint32_t *mask, const uint64_t *offsets, uint32_t *f_item, uint32_t *f_tid);

}  // namespace bm

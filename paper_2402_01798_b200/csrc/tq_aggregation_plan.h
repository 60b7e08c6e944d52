// How the aggregation cuts a row into tiles: plain arithmetic, shared by the launches and the kernels.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define TQ_PLAN_FN __host__ __device__ constexpr
#else
#define TQ_PLAN_FN constexpr
#endif

namespace tq {

constexpr int kDecThreads = 128;

// A unit is a run of elements decoded from one 32-bit "field": 8 / 16 / 32 elements = one packed word
// for 4 / 2 / 1 bits; for 3 bits 8 elements = 24 bits that start on a byte boundary and are cut out of
// two neighbouring words.  A thread owns U units, spaced one block apart, so that every
// load and every 256-bit store of a warp is contiguous, and keeps U * unit_elems (at most 32) accumulators in registers.
TQ_PLAN_FN int unit_elems(int bits) { return bits == 2 ? 16 : bits == 1 ? 32 : 8; }
TQ_PLAN_FN int unit_bytes(int bits) { return bits == 3 ? 3 : 4; }
TQ_PLAN_FN int most_units(int bits) { return 32 / unit_elems(bits); }      // of a thread with 32 accumulators
TQ_PLAN_FN uint32_t tile_bytes(int bits, int units) { return static_cast<uint32_t>(kDecThreads * units * unit_bytes(bits)); }   // one worker's, a multiple of 16
TQ_PLAN_FN uint64_t tiles_of(int bits, int units, uint64_t d) {            // each holds at least one element
    const uint64_t elems = static_cast<uint64_t>(kDecThreads) * units * unit_elems(bits);
    return (d + elems - 1) / elems;
}
// Bytes of a tile that starts `tile_off` bytes into a row of `row_bytes`; tile_off is inside the row.
TQ_PLAN_FN uint32_t tile_bytes_in_row(uint64_t row_bytes, uint64_t tile_off, uint32_t tile) {
    return row_bytes - tile_off < tile ? static_cast<uint32_t>(row_bytes - tile_off) : tile;
}

// Below this many tiles of 32 outputs per thread, two per SM, too few warps are in flight for the latency of a walk over the
// workers: the direct kernel takes one unit per thread (1 M x 64, 3 bits: 27.5 -> 17.3 us; 20 k x 64: 58 -> 7.9 us; 489 tiles, 2 M x
// 16: 10.8 us in the bulk form, 12.2 in the direct one).
constexpr uint64_t kTilesForBulk = 296;
// The fused update has as much to do after the walk as in it, and fewer registers per thread keep more of its loads in
// flight: one unit per thread up to this many tiles of 32 outputs per thread (4 M x 4: 18.6 -> 14.3 us, 11.2 M x 8: 39.9 -> 37.3;
// 25.6 M x 16, 6250 tiles: 102 us with one unit, 92.9 with two), beyond it two where a thread could have four (3 and 4 bits:
// 25.6 M x 16 96.6 -> 92.9 us, 50 M x 4 142 -> 130, 250 M x 4 684 -> 633).  With 64 workers the walk weighs more again: 3 M x 64
// takes 41.5 us with four units, 43.3 with two, 56 with one.
constexpr uint64_t kTilesForLongApply = 4096;
constexpr uint32_t kWorkersForShortApply = 32;

struct AggregationPlan {
    bool bulk;                 // the bulk-copy kernel, a block per tile; else the direct one
    int units;                 // per thread
    uint64_t blocks;
};
inline AggregationPlan plan_aggregation(int bits, uint64_t d, uint32_t n_workers, bool apply) {
    const int most = most_units(bits);
    const uint64_t tiles = tiles_of(bits, most, d);
    AggregationPlan p{tiles >= kTilesForBulk, most, 0};
    if (!p.bulk) p.units = 1;
    else if (apply && n_workers <= kWorkersForShortApply) p.units = tiles < kTilesForLongApply ? 1 : most > 2 ? 2 : most;
    p.blocks = tiles_of(bits, p.units, d);
    return p;
}

}  // namespace tq

// batch.cuh -- persistent kernel running many independent transforms of uneven
// sizes in one launch per field.
//
// The paper finds that short kernels run with sub-optimal launch parameters and
// calls for runtime autotuning (Section V-A); a server's batch holds many
// transforms too small to fill the GPU.  Here every pass of every transform is a
// segment of tiles; all tiles of all segments form one work list ordered by
// dependency level.  Resident blocks (one grid sized to the SM count) pull the
// next tile index from a device counter.  A segment may depend on an earlier one,
// the previous pass of the same transform; the block that claims a tile waits
// until that segment has retired all its tiles.  Because tiles are claimed in list
// order and every dependency points to an earlier position, the oldest unfinished
// tile can always run, so the scheme cannot deadlock however many blocks are
// resident.
//
// Every wait is bounded by `timeout_ns` (device global timer).  On expiry the
// block sets the launch's abort word and the sticky status word, and all blocks
// leave; the host reports ZKNTT_ETIMEOUT.
#pragma once
#include <cstdint>

#include "field.cuh"
#include "ntt_pass.cuh"

namespace zkntt {

constexpr int BATCH_MAX_SEGMENTS = 160;
constexpr uint32_t BATCH_THREADS = 256;
// blocks per SM the register budget is compiled for (80 registers a thread, which
// spill 112 to 208 bytes of stores: 64 uneven transforms of 2^10..2^20 in 1824 us;
// 64 registers 1926, 128 and two blocks, with nothing to cover a tile's loads, 2042)
#ifndef ZKNTT_BATCH_MIN_BLOCKS
#define ZKNTT_BATCH_MIN_BLOCKS 3
#endif
constexpr int BATCH_MIN_BLOCKS = ZKNTT_BATCH_MIN_BLOCKS;
// resident blocks per SM the tile-width policy counts as one wave
constexpr int BATCH_WAVE_BLOCKS = 3;
// widest batch tile, log2 elements (32 KiB, and up to 32 KiB of twiddle table: three
// blocks fit an SM's shared memory)
constexpr int BATCH_TILE_BITS = 10;
constexpr uint32_t BATCH_STATUS_TIMEOUT = 4u;  // == ZKNTT_ETIMEOUT

struct BatchSeg {
    PassArgs a;
    uint32_t first_item;  // index of the segment's first tile in the work list
    int32_t dep;          // segment that must be complete first (-1: none)
    uint32_t dep_tiles;   // its tiles
    uint32_t ntiles;      // tiles in this segment
    uint32_t job;         // index of the transform in the batch
    uint32_t signal;      // 1: last pass of its transform and completion words requested
};

struct BatchTable {
    uint32_t nseg;
    uint32_t total_items;
    unsigned long long timeout_ns;
    uint32_t *flags;      // per-transform completion words (may be null)
    uint32_t table_units; // 16-byte units of shared memory kept for the twiddle table
    uint32_t epoch;       // value written to flags[job] when the job completes
    BatchSeg seg[BATCH_MAX_SEGMENTS];
};

// passed by value as a kernel parameter (limit 32764 bytes)
static_assert(sizeof(BatchTable) <= 32000, "batch table exceeds the kernel parameter limit");

}  // namespace zkntt

// Host-side set-up shared by the entry points: once-per-device preparation and tensor-map construction.
#pragma once

#include <cuda.h>
#include <stdint.h>

namespace ais {

// Once per device (with that device current): architecture check, kernel attributes, the driver's tensor-map
// encoder.  Returns AIS_OK or AIS_ERR_DEVICE; *num_sms (may be NULL) receives the SM count.
int device_setup(int* num_sms);

// 2-D row-major tensor map (dim0 contiguous).  device_setup() must have succeeded before.
bool make_tmap(CUtensorMap* map, CUtensorMapDataType dtype, const void* base, uint64_t dim0, uint64_t dim1,
               uint64_t stride1_bytes, uint32_t box0, uint32_t box1, CUtensorMapSwizzle swz);

// The same matrix as [dim0 / 64][dim1][64] for boxes of four 64-column blocks x 64 rows (128-byte swizzle, one block after
// the other in shared memory).  dim0 has to be a multiple of 64, or the rows long enough to hold the rounded-up width.
bool make_tmap_blocks(CUtensorMap* map, const void* base, uint64_t dim0, uint64_t dim1, uint64_t stride1_bytes);

// How a forward or recompute pass over `rows` x `V` splits: row tiles per CTA and vocabulary ranges per unit of rows (at most
// `most`, or exactly `forced` if that is positive).
enum TileKind { kTileOne, kTileTwo, kTileBlock };   // 128 x 256 (lmhead.cu), 256 x 256 (lmhead_pair.cu), 256 x 128 (lmhead_fp8.cu)
struct PassPlan {
    bool two;          // kTileTwo
    int ranges;
    int unit_rows;     // rows of a unit
    int tile_cols;
    int parts() const { return 2 * ranges; }
};
PassPlan plan_kind(TileKind kind, int64_t rows, int V, int d, int most, int forced, double* cost);
// The better of kTileOne and kTileTwo.
PassPlan plan_pass(int64_t rows, int V, int d, int most, int forced);

// Bound of the kernels' device-side waits in clock ticks as set by ais_set_wait_cycles (0 = the kernels' default).
int64_t wait_cycles();

}  // namespace ais

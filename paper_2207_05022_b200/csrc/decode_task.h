// The unit of work of the weight decode, and the bounds it is held to.  Also compiled for the host by the tests.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include "host_device.h"

namespace sti {

// What one warp decodes of a weight tile: 4096 weights, 32 rows x 128 columns of a unit's matrix (64 x 64 when the
// matrix has 64 in-features).  Index streams are held re-tiled (see retile.h): the k 16-byte planes of the 32 lanes'
// quanta are stored plane-major, so that a warp reads each plane as one coalesced 512-byte line and every lane ends up
// with 128 consecutive indexes of one row.  Everything the warp needs to issue its loads stands in these 32 bytes: one
// memory round trip for the descriptor, one for planes, table and outliers together.
struct alignas(16) DecodeTask {
  const uint8_t* codes;     // device; first plane (uncompressed units: the fp32 rows, `out_val` bytes apart)
  uint32_t table;           // byte distances from `codes`: the unit's 2^bits fp32 centroids,
  uint32_t out_rc;          //   the task's outliers as (row << 16 | column) of the matrix,
  uint32_t out_val;         //   and their values
  uint16_t n_out;
  uint8_t bits;             // 2..6 or 32; 0 = no task
  uint8_t narrow;           // 1: 64 rows x 64 columns
  uint16_t row0, kcore0;    // place in the tile: first row, first group of eight columns
  uint32_t origin;          // (row << 16 | column) of the task's first weight in the matrix
};
static_assert(sizeof(DecodeTask) == 32, "two 16-byte loads");

// Row and column inside the task of the outlier at `rc` (row << 16 | column of the matrix); false if it is not one of the
// task's weights.  The lists come out of device memory that streamed layers overwrite in turn, so this is looked at where
// they are applied: a wrong entry is left out rather than stored somewhere else in shared memory.
STI_HOST_DEVICE bool outlier_place(const DecodeTask& t, uint32_t rc, uint32_t& row, uint32_t& col) {
  const uint32_t at = rc - t.origin;       // a column left of the task's borrows from the row: the column is then out of range
  row = at >> 16;
  col = at & 0xffffu;
  return (at & (t.narrow ? 0xffc0ffc0u : 0xffe0ff80u)) == 0;     // row < 64 and column < 64; row < 32 and column < 128
}

}  // namespace sti

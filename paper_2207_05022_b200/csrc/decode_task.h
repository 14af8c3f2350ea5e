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

// Tasks of a working buffer (expand.cu) name the first of their two 4 KB pieces in place of a row and a column group.
STI_HOST_DEVICE uint32_t expanded_at(const DecodeTask& t) { return t.row0 | static_cast<uint32_t>(t.kcore0) << 16; }

// Row and column inside the task of the outlier at `rc` (row << 16 | column of the matrix); false if it is not one of the
// task's weights.  The lists come out of device memory that streamed layers overwrite in turn, so this is looked at where
// they are applied: a wrong entry is left out rather than stored somewhere else in shared memory.
STI_HOST_DEVICE bool outlier_place(const DecodeTask& t, uint32_t rc, uint32_t& row, uint32_t& col) {
  const uint32_t at = rc - t.origin;       // a column left of the task's borrows from the row: the column is then out of range
  row = at >> 16;
  col = at & 0xffffu;
  return (at & (t.narrow ? 0xffc0ffc0u : 0xffe0ff80u)) == 0;     // row < 64 and column < 64; row < 32 and column < 128
}

// Whether a task stays inside its tile of n_rows x k_total and reads nothing but the `bytes` bytes of its unit at `unit`: looked
// at once for every task when a plan's tables are built, because the kernels follow a descriptor before anything else has
// arrived that they could hold it against.
inline bool task_in_bounds(const DecodeTask& t, uint32_t n_rows, uint32_t k_total, const uint8_t* unit, size_t bytes) {
  const uint32_t rows = t.narrow ? 64u : 32u, cols = t.narrow ? 64u : 128u;
  if (t.row0 + rows > n_rows || t.kcore0 * 8u + cols > k_total) return false;
  if (t.codes < unit || static_cast<size_t>(t.codes - unit) > bytes) return false;
  const size_t left = bytes - static_cast<size_t>(t.codes - unit);       // from `codes` to the unit's end
  auto holds = [&](size_t at, size_t n) { return at <= left && n <= left - at; };
  if (reinterpret_cast<uintptr_t>(t.codes) % 16 != 0) return false;
  if (t.bits == 32) return t.n_out == 0 && t.out_val % 16 == 0 && holds(0, static_cast<size_t>(rows - 1) * t.out_val + cols * 4u);
  if (t.bits < 2 || t.bits > 6) return false;
  const size_t outliers = static_cast<size_t>(t.n_out) * 4;
  return holds(0, 512u * t.bits) && t.table % 4 == 0 && holds(t.table, 4u << t.bits) &&
         t.out_rc % 4 == 0 && holds(t.out_rc, outliers) && t.out_val % 4 == 0 && holds(t.out_val, outliers);
}

}  // namespace sti

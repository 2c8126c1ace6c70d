// adi_tile_stage.h -- where the band step (adi_tile.cu) keeps a staged block
// in shared memory, and the byte offsets its row solves read from.  Plain
// constexpr arithmetic, so that the offsets of all threads can be enumerated
// on the host.
#pragma once

#include <stdint.h>

namespace adi {

constexpr int kTX = 224;              // columns a CTA solves
constexpr int kTH = 16;               // halo columns on either side
constexpr int kTB = 16;               // rows per block
constexpr int kTS = kTX + 2 * kTH;    // staged columns
constexpr int kTN = kTS / 2;          // threads: two rows (x phase) or two columns (y phase) each
constexpr int kTChunks = kTS / 16;    // chunks of 16 unknowns in a staged row
constexpr int kPanel = kTB * 128;     // bytes of a 32-column panel of a block
constexpr int kSlot = (kTS / 32) * kPanel;  // bytes of one staged block
constexpr int kUSlots = 3;            // slots of u^k, at the start of the stage

// First 16-byte unit of chunk c in row r of a block: the unit q of the chunk
// lies at the offset XOR 16 q (128-byte swizzle), row r + 8 lies 1024 bytes on.
constexpr uint32_t tile_unit(int r, int c) {
  return (uint32_t)((c >> 1) * kPanel + r * 128 + (((c & 1) * 64) ^ ((r & 7) << 4)));
}

// Offsets of rows r = xr and xr + 8 (h = 0, 1), chunk ch.  u^k's blocks are
// shifted by one row: rows r - 1, r, r + 1 of the block are at indexes r - 2,
// r - 1, r, the negative ones at the end of the block before, so that centre
// and above are relative to tile_row_base().
struct TileRow {
  uint32_t centre, above, below;  // u^k in rows r, r - 1 and r + 1 (below: relative to the block's slot)
  uint32_t left, right;           // the unknowns beside the chunk, relative as centre
};
constexpr TileRow tile_row(int xr, int ch) {
  TileRow t = {};
  t.centre = tile_unit(xr + 7, ch);
  t.above = tile_unit(xr + 6, ch);
  t.below = tile_unit(xr, ch);
  // The outermost chunks have no neighbour in the stage (the unknown that
  // would use it is zero): any word of the row does.
  t.left = ch > 0 ? (tile_unit(xr + 7, ch - 1) ^ 48u) + 12u : t.centre;
  t.right = ch < kTChunks - 1 ? tile_unit(xr + 7, ch + 1) : t.centre;
  return t;
}

// Base of the slot that holds row r - back of the block in slot cur (prev: the
// slot of the block before), for the offsets of TileRow; back = 0 (centre) or
// 1 (above).
constexpr uint32_t tile_row_base(uint32_t cur, uint32_t prev, int xr, int h, int back) {
  return h == 0 ? (xr >= 1 + back ? cur - 1024u : prev + 1024u) : cur;
}

}  // namespace adi

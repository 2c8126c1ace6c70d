"""Shared-memory offsets of the band step's row solves (csrc/adi_tile_stage.h),
enumerated on the host: every word a thread reads of u^k lies in the stage's
slots of u^k, and a unit that exists in the stage is the one that is meant."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "adi_tile_stage.h"
using namespace adi;
static int bad = 0;
// byte of column c, row r of a block
static uint32_t word(int r, int c) {
  return (uint32_t)((c >> 5) * kPanel + r * 128 + ((((c & 31) >> 2) ^ (r & 7)) << 4) + 4 * (c & 3));
}
static void check(uint32_t at, uint32_t bytes, const char* what, int slot, int tid, int h) {
  if (at > (uint32_t)(kUSlots * kSlot) - bytes && bad++ < 10)
    printf("%s of slot %d, thread %d, half %d: byte %d\n", what, slot, tid, h, (int)at);
}
static void same(uint32_t at, uint32_t want, const char* what, int slot, int tid, int h) {
  if (at != want && bad++ < 10)
    printf("%s of slot %d, thread %d, half %d: byte %d, not %d\n", what, slot, tid, h, (int)at, (int)want);
}
int main() {
  for (int slot = 0; slot < kUSlots; ++slot) {
    const uint32_t cur = slot * kSlot, prev = ((slot + kUSlots - 1) % kUSlots) * kSlot;
    for (int tid = 0; tid < kTN; ++tid) {
      const int xr = tid & 7, ch = tid >> 3;
      const TileRow t = tile_row(xr, ch);
      for (int h = 0; h < 2; ++h) {
        const uint32_t bc = tile_row_base(cur, prev, xr, h, 0), bu = tile_row_base(cur, prev, xr, h, 1);
        // row r of the block is index r - 1 of its slot, row -1 + k of it index 15 of the one before
        const int r = xr + 8 * h;
        auto row = [&](int k, int c) { return k >= 1 ? cur + word(k - 1, c) : prev + word(k + 15, c); };
        for (int q = 0; q < 4; ++q) {
          const uint32_t c = (bc + t.centre) ^ (16u * q), u = (bu + t.above) ^ (16u * q);
          const uint32_t d = ((cur + t.below) ^ (16u * q)) + 1024u * h;
          check(c, 16, "centre", slot, tid, h);
          check(u, 16, "above", slot, tid, h);
          check(d, 16, "below", slot, tid, h);
          same(c, row(r, 16 * ch + 4 * q), "centre", slot, tid, h);
          same(u, row(r - 1, 16 * ch + 4 * q), "above", slot, tid, h);
          same(d, row(r + 1, 16 * ch + 4 * q), "below", slot, tid, h);
        }
        check(bc + t.left, 4, "left", slot, tid, h);
        check(bc + t.right, 4, "right", slot, tid, h);
        if (ch > 0) same(bc + t.left, row(r, 16 * ch - 1), "left", slot, tid, h);
        if (ch < kTChunks - 1) same(bc + t.right, row(r, 16 * ch + 16), "right", slot, tid, h);
      }
    }
  }
  return bad != 0;
}
"""


def test_row_solves_read_inside_the_stage(tmp_path):
    src = tmp_path / "stage.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "stage")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2006_10142_gb300", "csrc"),
                    str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

"""The halo buffer of a slab face holds 2-byte populations ahead of FP32 side
planes and records: with an odd number of populations (one species or an odd
species count, an odd plane) those must still start on a word.  Every part at
a multiple of its element size, none overlapping, compiled and run here."""

import subprocess
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2004_11286_gb300" / "csrc"

PROGRAM = r"""
#include "lbm_halo.h"
#include <cstdio>
int main() {
  int bad = 0;
  for (int M = 1; M <= 8; ++M)
    for (size_t seg = 1; seg <= 200; ++seg)
      for (int prec = 0; prec < 4; ++prec) {
        const size_t es = prec == 0 ? 8 : (prec == 1 ? 4 : 2), ss = prec == 0 ? 8 : 4;
        const size_t rec = prec < 2 ? 0 : 2 * ((9 + M + 3) / 4 * 4), fields = (M + 2) * 27, nside = 20;
        const lbm::HaloLayout l = lbm::halo_layout(fields, seg, es, nside, ss, rec);
        bad += l.side % ss != 0 || l.rec % sizeof(float) != 0;
        bad += l.side < fields * seg * es || l.side >= fields * seg * es + ss;
        bad += l.rec != l.side + nside * seg * ss || l.bytes != l.rec + rec * seg * sizeof(float);
      }
  std::printf("%d\n", bad);
  return bad != 0;
}
"""


def test_every_part_is_aligned(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-I", str(CSRC), str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.strip() == "0"


def test_packing_takes_its_offsets_from_the_layout():
    api = (CSRC / "lbm_api.cu").read_text()
    move = api[api.index("static lbm_status halo_move"):]
    move = move[:move.index("\n}\n")]
    assert "b +=" not in move and "lay.side" in move and "lay.rec" in move

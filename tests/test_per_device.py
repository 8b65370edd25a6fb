"""What the launchers set up once (shared-memory limits, resident blocks) holds
for one device: a process with handles on two devices needs it on each.  The
table behind it is host code and is compiled and run here."""

import re
import subprocess
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2004_11286_gb300" / "csrc"

PROGRAM = r"""
#include "lbm_per_device.h"
#include <cstdio>
static lbm::PerDevice table;
int main() {
  int calls = 0, ok = 1;
  auto get = [&](int dev, int result) { return table.get(dev, [&] { ++calls; return result; }); };
  ok &= get(0, 7) == 7 && calls == 1;
  ok &= get(0, 8) == 7 && calls == 1;      // known
  ok &= get(1, 9) == 9 && calls == 2;      // another device
  ok &= get(2, 0) == 0 && calls == 3;      // failed: not remembered
  ok &= get(2, 5) == 5 && calls == 4;
  ok &= get(63, 1) == 1 && get(64, 2) == 2 && get(64, 3) == 3 && get(-1, 4) == 4 && calls == 8;
  std::printf("%d\n", ok);
  return !ok;
}
"""


def test_table_keeps_a_value_per_device(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-I", str(CSRC), str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.strip() == "1"


def test_launchers_keep_no_set_up_for_the_first_device_only():
    """No launcher sets a kernel's attributes behind a process-wide flag or in
    the initialiser of a static."""
    for f in list(CSRC.glob("*.cuh")) + list(CSRC.glob("*.cu")):
        code = re.sub(r"//[^\n]*", "", f.read_text())
        assert not re.search(r"static\s+(const\s+)?(bool|int)\s+\w+\s*=\s*(false|\[)", code), f.name

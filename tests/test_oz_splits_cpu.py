"""The split of K of the FP64 digit products (csrc/oz_splits.h), compiled for the host.

Each split's int32 sums must hold the largest sum that digits of magnitude 256 can give: (level + 1) 64 256^2 per piece,
level 7 of the skinny product included.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "oz_splits.h"
int main() {
  for (int level : {5, 7})
    for (int pieces = 1; pieces <= 4096; ++pieces)
      for (int64_t items : {1LL, 7LL, 152LL, 153LL, 4000LL, 100000LL}) {
        const int most = lrtei::oz::max_pieces(level);
        const int s = lrtei::oz::pick_splits(items, pieces, level == 5 ? 6.0 : 1.5, most);
        const long long per = (pieces + s - 1) / s;  // as the kernel cuts them
        if (s < 1 || per * (level + 1) * 64 * 65536 > 0x7FFFFFFFLL) {
          std::printf("level %d, %d pieces in %d splits of %lld\n", level, pieces, s, per);
          return 1;
        }
      }
  return 0;
}
"""


def test_int32_sums_hold_every_split(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "splits.cpp", tmp_path / "splits"
    src.write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2210_13069_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

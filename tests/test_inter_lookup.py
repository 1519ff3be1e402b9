"""The block table of an intermediate (csrc/engine.hpp, Inter::find): blocks
added after a lookup are found, indices outside the table are not read."""
import os
import subprocess

import paper_1902_08489_gb300 as td
from paper_1902_08489_gb300 import build

PROGRAM = r"""
#include "engine.hpp"
int main() {
  tdmps::Inter t;
  if (t.find(0, -1, 0, 0) != -1) return 1;
  t.add(0, -1, 0, 2, 1, 1, 1);
  if (t.find(0, -1, 0, 2) != 0 || t.find(0, -1, 0, 1) != -1) return 2;
  t.add(3, 2, 1, 4, 1, 1, 1);
  if (t.find(3, 2, 1, 4) != 1 || t.find(0, -1, 0, 2) != 0) return 3;
  if (t.find(-1, -1, 0, 0) != -1 || t.find(0, -1, -1, 0) != -1) return 4;
  if (t.find(0, 4, 0, 0) != -1 || t.find(0, -2, 0, 0) != -1 || t.find(4, 0, 0, 0) != -1) return 5;
  t.add(3, 2, 1, 5, 1, 1, 1);
  try {
    t.find(3, 2, 1, 5);
  } catch (const tdmps::Error&) {
    return 0;
  }
  return 6;
}
"""


def test_lookup_follows_the_blocks(tmp_path):
    td.lib()
    src, exe = tmp_path / "lookup.cpp", tmp_path / "lookup"
    src.write_text(PROGRAM)
    inc = [os.path.dirname(os.path.dirname(build.nvcc())) + "/include", build.SRC,
           os.path.join(build.HERE, "..", "include")]
    subprocess.run(["g++", "-std=c++17", str(src), "-o", str(exe), *["-I" + i for i in inc],
                    build.LIB, "-Wl,-rpath," + build.OUT], check=True)
    assert subprocess.run([str(exe)]).returncode == 0

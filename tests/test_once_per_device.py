"""Kernel attributes are set once per device, not once per process (the bookkeeping, with devices and a setter made up here)."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_19324_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "once_per_device.h"
int main() {
  rsd::OncePerDevice a, b;
  int calls[3] = {0, 0, 0};
  auto on = [&](rsd::OncePerDevice& o, int dev, int slot, int result) { return o.run(dev, [&] { ++calls[slot]; return result; }); };
  int bad = 0;
  for (int i = 0; i < 3; ++i) bad += on(a, 0, 0, 0) != 0;      // first device: once
  bad += calls[0] != 1;
  for (int i = 0; i < 3; ++i) bad += on(a, 1, 1, 0) != 0;      // the second device has its own turn
  bad += calls[1] != 1;
  bad += on(a, 0, 0, 0) != 0 || calls[0] != 1;
  bad += on(b, 0, 2, 7) != 7;                                  // a failure is returned and tried again
  bad += on(b, 0, 2, 0) != 0 || calls[2] != 2;
  bad += on(b, 0, 2, 7) != 0 || calls[2] != 2;
  calls[2] = 0;
  for (int i = 0; i < 2; ++i) bad += on(b, 64, 2, 0) != 0;     // beyond what is noted: every time
  bad += on(b, 63, 2, 0) != 0;
  bad += on(b, 63, 2, 0) != 0 || calls[2] != 3;
  std::printf("%d\n", bad);
  return bad;
}
"""


def test_once_for_every_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.strip() == "0"


def test_no_launch_site_sets_attributes_once_per_process():
    """`static x = cudaFuncSetAttribute(...)` and `if (!configured)` run on the first device only."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"cudaFuncSetAttribute", text):
            before = text[max(0, m.start() - 160):m.start()]
            assert not re.search(r"static [^;]*$|if \(!?configured[^;]*$", before), (name, text[:m.start()].count("\n") + 1)

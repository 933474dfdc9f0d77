"""What the library finds out once per device (launch limits, function
attributes) is found out on every device: the second one does not take over
the first one's answer.  The cache is plain C++, so this runs without a GPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "per_device.h"
int main() {
  static bo::PerDevice p;
  int asked = 0;
  auto on = [&](int device, int answer) {
    return p.get(device, [&] { ++asked; return answer; }) == answer;
  };
  bool ok = on(0, 16) && on(0, 16) && asked == 1;       // once per device
  ok = ok && on(1, 8) && asked == 2 && on(0, 16) && on(1, 8) && asked == 2;
  ok = ok && on(2, 0) && on(2, 0) && asked == 3;        // zero is an answer too
  ok = ok && on(bo::PerDevice::kMax, 4) && on(bo::PerDevice::kMax, 2) && asked == 5;  // beyond the table: asked again
  return ok ? 0 : 1;
}
"""


def test_every_device_is_asked_once(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I",
                    os.path.join(ROOT, "paper_1606_00556_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0

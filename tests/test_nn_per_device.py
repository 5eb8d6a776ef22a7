"""Kernel attributes of the network's launches are set once per device, not once per
process (host code, compiled and run here)."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_02185_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "nn_per_device.h"
int main() {
  static gbnn_tc::PerDevice once;
  int calls = 0;
  auto find = [&] { return ++calls; };
  int out[9], n = 0;
  for (int dev : {0, 0, 1, 1, 0, 63, 64, 64, -1}) out[n++] = once.get(dev, find);
  for (int i = 0; i < n; ++i) std::printf("%d ", out[i]);
  static gbnn_tc::PerDevice failing;
  int tries = 0;
  auto late = [&] { return ++tries < 3 ? -1 : 7; };
  for (int i = 0; i < 4; ++i) std::printf("%d ", failing.get(2, late));
  std::printf("%d", tries);
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "p.cc", tmp_path / "p"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    # found on devices 0, 1, 63; each time past the last; a failure is tried again
    assert out.split() == ["1", "1", "2", "2", "1", "3", "4", "5", "6", "-1", "-1", "7", "7", "3"]


def test_every_launch_asks_per_device():
    for name in ("nn_tc.cu", "nn_rows.cuh"):
        text = open(os.path.join(CSRC, name)).read()
        for once_per_process in ("static int per_sm", "static int sms", "static bool prepared"):
            assert once_per_process not in text, (name, once_per_process)

"""Kernel settings that hold per device (csrc/per_device.h), driven on the host: each device of a process gets
its own, once, a failed setting is tried again, and threads that meet there all find it set."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1212_1397_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
int main() {
  helm6::OncePerDevice once;
  int calls[70] = {};
  auto set = [&](int d, bool good) { return once(d, [&] { ++calls[d < 0 ? 69 : d]; return good; }); };
  printf("%d", set(0, true));
  printf("%d", set(0, true));
  printf("%d", set(1, false));  // a second device is not taken for the first
  printf("%d", set(1, true));
  printf("%d", set(1, true));
  printf("%d", set(63, true));
  printf("%d", set(64, true));  // beyond the 64 that are remembered, and unknown: set each time
  printf("%d", set(64, true));
  printf("%d", set(-1, true));
  printf("%d", set(-1, true));
  printf(" %d %d %d %d %d\n", calls[0], calls[1], calls[63], calls[64], calls[69]);
  helm6::OncePerDevice shared;
  std::atomic<int> missing{0};
  std::atomic<unsigned> have{0};
  std::vector<std::thread> t;
  for (int i = 0; i < 8; ++i)
    t.emplace_back([&, i] {
      const int d = i & 3;
      if (!shared(d, [&] { have.fetch_or(1u << d); return true; }) || !(have.load() >> d & 1u)) missing++;
    });
  for (auto& x : t) x.join();
  printf("%d\n", missing.load());
}
"""


def test_each_device_once(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no C++ compiler")
    src = tmp_path / "per_device.cpp"
    src.write_text(SOURCE)
    exe = str(tmp_path / "per_device")
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
    assert out[:2] == ["1101111111 1 2 1 2 2", "0"]


def test_no_setting_is_kept_for_the_whole_process():
    """The kernels' attributes are set nowhere but behind a per-device flag."""
    for name in sorted(os.listdir(CSRC)):
        if name.endswith(".cu"):
            text = open(os.path.join(CSRC, name)).read()
            if "cudaFuncSetAttribute" in text:
                assert "OncePerDevice" in text, name
                for word in ("static bool done", "static int done", "static bool configured"):
                    assert word not in text, (name, word)

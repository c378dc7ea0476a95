"""PerDevice (csrc/qf_per_device.h): set-up runs once on each device, not once in the process."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2211_10185_gb300", "csrc")
PROGRAM = """
#include <stdio.h>
#include <thread>
#include <vector>
#include "qf_per_device.h"
int main() {
  qf::PerDevice done;
  std::atomic<int> calls[3] = {};
  std::vector<std::thread> t;
  std::atomic<int> bad{0};
  for (int k = 0; k < 24; ++k)
    t.emplace_back([&, k] {
      const int dev = k % 3;
      for (int i = 0; i < 100; ++i)
        if (done.ready(dev, [&] { return ++calls[dev], dev != 1; }) != (dev != 1)) ++bad;
    });
  for (auto& x : t) x.join();
  printf("%d %d %d %d\\n", calls[0].load(), calls[1].load(), calls[2].load(), bad.load());
  return 0;
}
"""


def test_set_up_once_per_device(tmp_path):
    cxx = shutil.which("g++") or pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cc", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["1", "1", "1", "0"]


def test_no_kernel_attribute_is_set_once_per_process():
    """Every launcher that sets function attributes goes through PerDevice."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        if "done.ready(" not in text:
            assert "cudaFuncSetAttribute" not in text, name
        assert "static bool attr" not in text and "static const bool ready" not in text, name

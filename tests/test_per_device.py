"""Set-up that holds for one device (a kernel's limit of dynamic shared memory) is
done for each device that a process uses, by whichever thread comes first, and a
failure is tried again: csrc/per_device.h by itself, and its use by every launch."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_13308_gb300", "csrc")

PROGRAM = r'''
#include <cassert>
#include <thread>
#include <vector>
#include "per_device.h"
int main() {
  vqmc::OncePerDevice once;
  std::atomic<int> made[8] = {};
  int fails = 1, odd = 0;
  // a failure is returned and tried again
  assert(once(3, [&] { return fails-- > 0 ? 7 : 0; }) == 7);
  assert(once(3, [&] { ++made[3]; return 0; }) == 0);
  assert(once(3, [&] { return 9; }) == 0 && made[3] == 1);
  // every device has its own; nobody returns before its device is set up
  std::vector<std::thread> threads;
  for (int t = 0; t < 16; ++t)
    threads.emplace_back([&, t] {
      for (int i = 0; i < 1000; ++i) {
        const int d = (t + i) % 3;
        assert(once(d, [&] { ++made[d]; return 0; }) == 0 && made[d] >= 1);
      }
    });
  for (auto& t : threads) t.join();
  for (int d = 0; d < 3; ++d) assert(made[d] <= 16);
  // devices beyond the table are set up on every call
  for (int i = 0; i < 2; ++i) assert(once(256, [&] { ++odd; return 0; }) == 0 && once(-1, [&] { ++odd; return 0; }) == 0);
  assert(odd == 4);
}
'''


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-UNDEBUG", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    subprocess.run([str(exe)], check=True, timeout=60)


def test_no_process_wide_flag_guards_a_launch():
    """No file keeps a flag of its own for what was set on one device."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.search(r"^\s*(static\s+)?bool\s+g_\w+\s*=", text, re.M), path

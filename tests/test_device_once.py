"""A kernel's shared memory limit belongs to one device: what raises it does so
once on every device that launches the kernel, not once per process.  The
bookkeeping (csrc/device_once.h) needs no GPU: a small host program runs it over
made-up device numbers."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_08340_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include <thread>
#include <vector>
#include "device_once.h"
int main() {
  static oprag::DeviceOnce once;
  int calls[128] = {0}, fail_on = 2;
  auto use = [&](int dev) { return once.run(dev, [&] { ++calls[dev]; return dev == fail_on ? 7 : 0; }); };
  for (int round = 0; round < 3; ++round)
    for (int dev : {0, 1, 63, 2, 64, 127}) {
      const int rc = use(dev);
      if (rc != (dev == fail_on ? 7 : 0)) return 1;
    }
  fail_on = -1;                      // a failure is not remembered as done
  if (use(2) != 0 || use(2) != 0) return 2;
  std::printf("%d %d %d %d %d %d\n", calls[0], calls[1], calls[63], calls[2], calls[64], calls[127]);
  oprag::DeviceOnce shared;          // each device's first user does the work itself
  std::vector<std::thread> pool;
  int done[8] = {0};
  for (int d = 0; d < 8; ++d)
    pool.emplace_back([&, d] { for (int i = 0; i < 1000; ++i) shared.run(d, [&] { ++done[d]; return 0; }); });
  for (auto& t : pool) t.join();
  for (int d = 0; d < 8; ++d) if (done[d] != 1) return 3;
  return 0;
}
"""


def test_work_is_done_once_on_every_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    (tmp_path / "once.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "once")
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(tmp_path / "once.cpp"),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0
    # the failing device 2 tried on each call, then once more; 64 and 127 each time
    assert r.stdout.split() == ["1", "1", "1", "4", "3", "3"]


def test_no_limit_is_raised_once_per_process():
    for name in os.listdir(CSRC):
        text = open(os.path.join(CSRC, name)).read()
        assert not re.search(r"static\s+bool\b", text), f"{name}: a process-wide switch"

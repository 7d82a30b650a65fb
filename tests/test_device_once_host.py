"""What a launcher settles once belongs to a device, not to the process.

A kernel's dynamic shared-memory limit has to be raised on every device that runs it (a network or a
context takes a device number). The memo behind it is compiled here without CUDA: an action runs once
per device, again after a failure, and from several threads at the same time; and every launcher goes
through it."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2412_10167_gb300", "csrc")

PROGRAM = r"""
#include <cassert>
#include <thread>
#include <vector>
#include "mw3_device.h"
int main() {
  mw3::OncePerDevice once;
  int calls[70] = {};
  auto set = [&](int dev, int status) { return once.run(dev, [&] { ++calls[dev]; return status; }); };
  assert(set(0, 0) == 0 && set(0, 0) == 0 && calls[0] == 1);
  assert(set(1, 0) == 0 && calls[1] == 1);                  // another device: the action again
  assert(set(63, 7) == 7 && set(63, 0) == 0 && set(63, 9) == 0 && calls[63] == 2);   // after a failure
  assert(set(64, 0) == 0 && set(64, 0) == 0 && calls[64] == 2);   // beyond the memo: every time
  mw3::IntPerDevice value;
  int computed = 0;
  auto get = [&](int dev) { return value.get(dev, [&] { ++computed; return 10 + dev; }); };
  assert(get(0) == 10 && get(0) == 10 && get(5) == 15 && get(5) == 15 && computed == 2);
  assert(get(64) == 74 && get(-1) == 9 && computed == 4);
  mw3::OncePerDevice shared;
  std::atomic<int> done{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&, t] {
      for (int i = 0; i < 1000; ++i) assert(shared.run((t + i) % 64, [&] { ++done; return 0; }) == 0);
    });
  for (auto& t : ts) t.join();
  assert(done >= 64 && done <= 64 * 8);
  return 0;
}
"""


def test_actions_run_once_per_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    subprocess.run([str(exe)], check=True, timeout=60)


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_launchers_keep_no_process_wide_device_state(name):
    text = open(os.path.join(CSRC, name)).read()
    assert "cudaFuncSetAttribute" not in text        # through allow_smem, once per device
    assert not re.search(r"\bstatic\s+(bool|int)\s+\w+(\[\d+\])?\s*(=|,|;)", text)

"""Set-up that belongs to a device is done on each one (device_once.h), by the host compiler.

A kernel's shared-memory attribute is set per device; remembered per process, the
second device of a process never gets it and its handles are refused.
"""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2306_07603_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "device_once.h"
int main() {
  static ifd::DeviceOnce once;
  std::atomic<int> calls[3] = {};
  auto use = [&](int device, bool works) {
    return once(device, [&] { ++calls[device]; return works; });
  };
  std::vector<std::thread> all;
  for (int t = 0; t < 16; ++t) all.emplace_back([&, t] { use(t & 1, true); });
  for (auto &t : all) t.join();
  const bool failed = !use(2, false), again = use(2, true), kept = use(2, false);
  std::printf("%d %d %d %d%d%d\n", calls[0].load(), calls[1].load(), calls[2].load(), failed, again, kept);
}
"""


def test_each_device_is_set_up_once(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    (tmp_path / "once.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "once")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, "-o", exe, str(tmp_path / "once.cpp")],
                   check=True)
    assert subprocess.check_output([exe], text=True).strip() == "1 1 2 111"


def test_kernel_attributes_are_set_through_it():
    text = open(os.path.join(CSRC, "fused.cuh")).read()
    body = re.search(r"configure_nt\(\) \{(.*?)\n\}", text, re.S).group(1)
    assert "DeviceOnce" in body and "cudaGetDevice" in body and "static bool" not in body

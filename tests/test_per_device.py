"""Values kept per device (csrc/per_device.h), compiled for the host: each
device's is made when that device first asks, once however many threads do, and
is not another's.  What is kept this way (shared memory limits of kernels, SM
counts) is never kept once per process."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_17337_gb300", "csrc")

PROGRAM = r"""
#include <atomic>
#include <thread>
#include <vector>
#include "per_device.h"
int main() {
  static ibm::PerDevice<int> v;
  static std::atomic<int> made[80];
  auto ask = [](int d) { return v.get(d, [d] { return 100 * ++made[d] + d; }); };
  std::vector<std::thread> ts;
  std::atomic<int> bad{0};
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&] {
      for (int n = 0; n < 3; ++n)
        for (int d = 0; d < 64; ++d)
          if (ask(d) != 100 + d) ++bad;
    });
  for (auto& t : ts) t.join();
  for (int d = 0; d < 64; ++d)
    if (made[d] != 1) return 1;
  if (bad) return 2;
  if (ask(70) != 170 || ask(70) != 270) return 3;  // beyond the table: made on every use
  return 0;
}
"""


def test_each_device_has_its_own_value(tmp_path):
    cxx = os.environ.get("CXX") or shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "per_device.cpp", tmp_path / "per_device"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0


def test_device_attributes_are_not_kept_once_per_process():
    """Function bodies that set a kernel's attribute or ask a device's hold no
    `static bool` and no single `std::once_flag`."""
    for fn in sorted(os.listdir(CSRC)):
        if not fn.endswith(".cu"):
            continue
        src = open(os.path.join(CSRC, fn)).read()
        for body in re.split(r"\n}", src):
            if "cudaFuncSetAttribute(" in body or "cudaDeviceGetAttribute(" in body:
                assert not re.search(r"static (const )?(bool|int) \w+ ?[=;]|static std::once_flag \w+;", body), (fn, body[-400:])

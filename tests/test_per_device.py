"""Values kept per GPU by the launch code (csrc/per_device.h), compiled here with a
stand-in for the device calls: every device is set up at its own first use, once also
under several threads, and an error is returned and not kept (CPU only)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_17033_gb300", "csrc")

PROBE = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
enum Err { OK = 0, BAD = 101, FAULT = 7 };
int fills[4];
int main() {
  static sp2::PerDevice kept;
  auto use = [&](int dev, int* v) {
    return kept.get(dev, BAD, v, [&](int* n) { ++fills[dev]; *n = 10 + dev; return OK; });
  };
  std::vector<std::thread> t;
  for (int i = 0; i < 8; ++i)
    t.emplace_back([&, i] { int v; for (int k = 0; k < 1000; ++k) use(i % 2, &v); });
  for (auto& x : t) x.join();
  int v0 = 0, v1 = 0, v2 = 0, w = 0;
  if (use(0, &v0) != OK || use(1, &v1) != OK) return 1;
  if (v0 != 10 || v1 != 11 || fills[0] != 1 || fills[1] != 1) return 2;
  if (kept.get(2, BAD, &v2, [&](int*) { return FAULT; }) != FAULT) return 3;
  if (use(2, &v2) != OK || v2 != 12) return 4;
  if (kept.get(-1, BAD, &w, [&](int*) { return OK; }) != BAD) return 5;
  if (kept.get(sp2::kMaxDevices, BAD, &w, [&](int*) { return OK; }) != BAD) return 6;
  return 0;
}
"""


def test_each_device_is_set_up_once(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run([cxx, "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0


@pytest.mark.parametrize("name", ["gemm_tc.cu", "gemm_dig.cu"])
def test_launch_code_keeps_no_device_value_for_the_process(name):
    """The resident counts, and the shared-memory limits set with them, are per device."""
    src = open(os.path.join(CSRC, name)).read()
    assert src.count("static PerDevice kept;") == 1
    assert "static int resident" not in src and "static int n = 0" not in src

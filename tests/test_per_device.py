"""Values kept per device on the host (shared-memory limits, cluster occupancy): set up again for another
device, not kept when the set-up failed, safe from several threads, and asked every time past the table.
The header is plain C++ and is compiled here with the host compiler (devices are numbers).
"""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

SRC = r"""
#include "per_device.h"
#include <cstdio>
#include <thread>
#include <vector>
int main() {
  static chem::PerDevice p;
  int calls = 0;
  auto set = [&](int v) { return [&calls, v] { ++calls; return v; }; };
  if (p.get(0, set(3)) != 3 || p.get(0, set(9)) != 3 || calls != 1) return 1;   // once
  if (p.get(1, set(5)) != 5 || p.get(0, set(9)) != 3 || calls != 2) return 2;   // again for another device
  if (p.get(2, set(0)) != 0 || p.get(2, set(-1)) != -1 || p.get(2, set(4)) != 4 || calls != 5) return 3;  // not kept
  if (p.get(64, set(7)) != 7 || p.get(64, set(8)) != 8 || p.get(-1, set(6)) != 6 || calls != 8) return 4;
  static chem::PerDevice q;
  std::vector<std::thread> t;
  int bad[8] = {};
  for (int i = 0; i < 8; ++i)
    t.emplace_back([&bad, i] {
      for (int r = 0; r < 20000; ++r)
        if (q.get(r % 64, [r] { return 1 + r % 64; }) != 1 + r % 64) bad[i] = 1;
    });
  for (auto& x : t) x.join();
  for (int b : bad) if (b) return 5;
  std::puts("ok");
  return 0;
}
"""


def test_per_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I",
                    os.path.join(ROOT, "paper_2402_18858_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.returncode


def test_no_flag_per_process_in_the_launchers():
    """A static flag would skip the set-up on a second device."""
    d = os.path.join(ROOT, "paper_2402_18858_gb300", "csrc")
    for name in sorted(os.listdir(d)):
        text = open(os.path.join(d, name)).read()
        assert "static bool" not in text, name

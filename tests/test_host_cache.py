"""The launchers' per-device caches (host_cache.h): a failed question is not kept,
devices are kept apart, and threads that ask at the same time never see a value
before it is known.  Compiled with the host compiler; no GPU needed."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

PROGRAM = r"""
#include "host_cache.h"
#include <cstdio>
#include <thread>
#include <vector>
#define CHECK(x) do { if (!(x)) { std::printf("failed: %s\n", #x); return 1; } } while (0)
int main() {
  ccm::DeviceCache c;
  int asked = 0;
  CHECK(c.get(0, 1, [&] { ++asked; return 0; }) == 1);   // failed: the fallback, this time only
  CHECK(c.get(0, 1, [&] { ++asked; return -3; }) == 1);
  CHECK(c.get(0, 1, [&] { ++asked; return 6; }) == 6);
  CHECK(c.get(0, 1, [&] { ++asked; return 9; }) == 6 && asked == 3);
  CHECK(c.get(1, 1, [] { return 4; }) == 4);              // another device's own
  CHECK(c.get(0, 1, [] { return 9; }) == 6);
  for (int dev : {-1, 1000}) {                            // outside the table: asked every time
    CHECK(c.get(dev, 1, [] { return 5; }) == 5);
    CHECK(c.get(dev, 1, [] { return 0; }) == 1);
  }
  for (int round = 0; round < 200; ++round) {
    ccm::DeviceCache d;
    std::vector<int> got(8);
    std::vector<std::thread> t;
    for (int i = 0; i < 8; ++i)
      t.emplace_back([&, i] { got[i] = d.get(2, 1, [] { std::this_thread::yield(); return 7; }); });
    for (auto& x : t) x.join();
    for (int v : got) CHECK(v == 7);
  }
  return 0;
}
"""


def test_device_cache(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "cache.cpp", tmp_path / "cache"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O2", "-pthread", "-I",
                    os.path.join(ROOT, "paper_1303_0270_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout

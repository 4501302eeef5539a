"""Launch state is kept per device, and threads may fill it together: the
number of CTAs that a device holds, and with it the dynamic shared memory that
a kernel has been allowed there, is looked up on each device's first use."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_03092_gb300", "csrc")

PROGRAM = r"""
#include "per_device.h"

#include <cstdio>
#include <thread>
#include <vector>

#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }

static int finds[66];

int main() {
  static s2d::PerDevice state;
  auto use = [](int dev) { return state.get(dev, [dev] { finds[dev]++; return 100 + dev; }); };
  // each device has its own number, found once
  for (int round = 0; round < 3; round++)
    for (int dev = 0; dev < 64; dev++) CHECK(use(dev) == 100 + dev);
  for (int dev = 0; dev < 64; dev++) CHECK(finds[dev] == 1);
  // a device out of range is answered, and not kept
  CHECK(use(64) == 164 && use(64) == 164 && finds[64] == 2);
  // a failure is not kept
  static s2d::PerDevice failing;
  int tries = 0;
  auto find = [&] { return ++tries == 2 ? 7 : 0; };
  CHECK(failing.get(1, find) == 0 && failing.get(1, find) == 7 && failing.get(1, find) == 7 && tries == 2);
  // threads on alternating devices
  static s2d::PerDevice shared;
  static int wrong[8];
  std::vector<std::thread> threads;
  for (int t = 0; t < 8; t++)
    threads.emplace_back([t] {
      for (int i = 0; i < 20000; i++) {
        const int dev = (t + i) % 5;
        wrong[t] += shared.get(dev, [dev] { return 10 + dev; }) != 10 + dev;
      }
    });
  for (auto& t : threads) t.join();
  for (int t = 0; t < 8; t++) CHECK(wrong[t] == 0);
  return 0;
}
"""


def test_numbers_per_device(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    (tmp_path / "t.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-pthread", "-I", CSRC, "-o", exe,
                    str(tmp_path / "t.cpp")], check=True, timeout=300)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout


def test_no_unguarded_launch_state():
    """No function keeps a plain static number between calls: it would be one
    device's for all, and written by several threads at once."""
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            code = re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)
        plain = re.findall(r"^\s+static (?:unsigned |signed )?(?:int|bool|long|size_t|u?int\d+_t)\b[^()]*?[;=]", code,
                           flags=re.M)
        assert plain == [], (name, plain)

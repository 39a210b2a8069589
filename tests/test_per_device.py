"""Kernel attributes are set on every device that a process launches on (csrc/per_device.h), with host code only."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2010_13213_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include <thread>
#include <vector>
#include "per_device.h"
static int fail(int line) { printf("line %d\n", line); return 1; }
#define CHECK(x) if (!(x)) return fail(__LINE__)
int main() {
  static lgf::PerDevice p;
  int calls = 0;
  auto ok = [&] { ++calls; return true; };
  p.run(0, ok), p.run(0, ok);
  CHECK(calls == 1);                        // once on a device
  p.run(1, ok), p.run(63, ok), p.run(0, ok), p.run(1, ok), p.run(63, ok);
  CHECK(calls == 3);                        // and once on every other
  p.run(2, [&] { ++calls; return false; });
  p.run(2, ok), p.run(2, ok);
  CHECK(calls == 5);                        // a failure is not remembered
  p.run(64, ok), p.run(64, ok), p.run(-1, ok);
  CHECK(calls == 8);                        // beyond the table: every time
  for (int round = 0; round < 200; ++round) {  // after run() the work is done, whichever thread did it
    lgf::PerDevice q;
    std::atomic<int> set{0};
    std::atomic<bool> missing{false};
    std::vector<std::thread> t;
    for (int i = 0; i < 4; ++i)
      t.emplace_back([&] {
        q.run(3, [&] { set.fetch_add(1); return true; });
        if (set.load() < 1) missing = true;
      });
    for (auto &x : t) x.join();
    CHECK(!missing);
  }
  return 0;
}
"""


def test_once_per_device(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_no_attribute_is_remembered_per_process():
    """Every launch site goes through the per-device record, or sets the attribute on each call."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for word in ("static bool attr", "static bool done", "call_once"):
            assert word not in text, (name, word)

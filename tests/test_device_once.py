"""Kernel attributes (the shared-memory limit) are set once on each device, not once per
process: the helper that remembers it, compiled alone, and that every launcher goes
through it."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_03345_gb300", "csrc")

PROGRAM = r"""
#include "device_once.h"
#include <thread>
#include <vector>
int main() {
  static fwi::DeviceOnce once, other;
  for (int d : {0, 1, 63}) {
    if (once.done(d)) return 1;        // a device set up leaves the next one to do
    once.mark(d);
    if (!once.done(d)) return 2;
  }
  if (once.done(2) || other.done(0)) return 3;
  for (int d : {-1, 64, 1000}) {       // never remembered: set up each time
    once.mark(d);
    if (once.done(d)) return 4;
  }
  std::vector<std::thread> t;
  for (int d = 0; d < 64; ++d) t.emplace_back([d] { other.mark(d); });
  for (auto& x : t) x.join();
  for (int d = 0; d < 64; ++d)
    if (!other.done(d)) return 5;
  return 0;
}
"""


def test_each_device_is_set_up(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_every_launcher_uses_it():
    calls = {}
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        calls[f] = len(re.findall(r"cudaFuncSetAttribute\(", text))
        assert "static bool" not in text, f
    assert {f: n for f, n in calls.items() if n} == {"fwi_internal.cuh": 2}

"""A kernel's limit of dynamic shared memory is kept by the CUDA runtime per device and the last value set
counts: the library raises it once per device and never lowers it, from several host threads too.  Compiled
and run on the host with a stand-in for cudaFuncSetAttribute."""
import os
import re
import subprocess

from ._util import ROOT

CSRC = os.path.join(ROOT, "paper_2311_12134_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include "internal.h"
using namespace lsms;
static std::atomic<int> value[4], calls[4];
static int set(int dev, int bytes) { value[dev] = bytes; ++calls[dev]; return LSMS_OK; }
int main() {
  static SmemLimit a, b;
  for (int rep = 0; rep < 2; ++rep)
    for (int dev = 0; dev < 2; ++dev)
      if (a.raise(dev, 70000, [&] { return set(dev, 70000); })) return 1;
  if (value[0] != 70000 || value[1] != 70000 || calls[0] != 1 || calls[1] != 1) return 2;  // each device, once
  std::thread t[8];
  for (int i = 0; i < 8; ++i)
    t[i] = std::thread([i] {
      for (int k = 0; k < 1000; ++k) {
        const int bytes = 50000 + 8 * ((k * 37 + i * 11) % 1000);
        b.raise(2, bytes, [&] { return set(2, bytes); });
        if (value[2] < bytes) std::_Exit(3);  // a launch of `bytes` would be refused
      }
    });
  for (auto& x : t) x.join();
  if (b.raise(3, 60000, [] { return -2; }) != -2) return 4;        // a failure is passed on
  if (b.raise(3, 60000, [&] { return set(3, 60000); }) || calls[3] != 1) return 5;  // and tried again
  return b.raise(64, 1, [] { return -7; }) == -7 ? 0 : 6;
}
"""


def test_limits_are_raised_once_per_device(tmp_path):
    src, exe = tmp_path / "limit.cpp", tmp_path / "limit"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_every_kernel_asks_per_device():
    for name in os.listdir(CSRC):
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        assert name == "common.cuh" or "cudaFuncSetAttribute" not in text, name
        assert not re.search(r"static\s+(bool|size_t|int)\s+\w*attr", text), name

"""Steps that belong to a device (kernel attributes) are done once per device, again for the next
device of the same thread, and again after a failure; every launcher that raises a kernel's
shared-memory limit goes through that bookkeeping (a small host program, no GPU).
"""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_16850_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include "device_once.h"
int main() {
  deer::DeviceOnce once, other;
  int calls[80] = {};
  auto step = [&](int dev, int status) {
    return once.ensure(dev, [&] { ++calls[dev]; return status; });
  };
  bool ok = step(0, 7) == 7 && calls[0] == 1;        // a failure is reported
  ok = ok && step(0, 0) == 0 && calls[0] == 2;       // and tried again
  ok = ok && step(0, 0) == 0 && calls[0] == 2;       // done
  ok = ok && step(1, 0) == 0 && calls[1] == 1;       // another device, the same thread
  ok = ok && step(1, 0) == 0 && calls[1] == 1 && step(0, 0) == 0 && calls[0] == 2;
  ok = ok && step(63, 0) == 0 && step(63, 0) == 0 && calls[63] == 1;
  ok = ok && step(64, 0) == 0 && step(64, 0) == 0 && calls[64] == 2;  // past the table
  std::thread([&] { ok = ok && step(1, 0) == 0 && calls[1] == 1; }).join();
  int n = 0;
  ok = ok && other.ensure(1, [&] { ++n; return 0; }) == 0 && n == 1;  // another kernel
  std::puts(ok ? "ok" : "wrong");
  return ok ? 0 : 1;
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.strip() == "ok"


def test_attributes_are_set_per_device():
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"cudaFuncSetAttribute\(", text):
            before = text[max(0, m.start() - 120):m.start()]
            assert ".ensure(dev" in before, (name, text[m.start():m.start() + 80])

"""Values that belong to one device are found once per device (per_device.h): a kernel's shared-memory limit set on
one device says nothing about another, and two threads may make the first call together."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1710_08231_gb300", "csrc")

_PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
int main() {
  gp::PerDevice p;
  int kernel[2], made = 0, v = 0;
  auto give = [&](int x) { return [&made, x](int *out) { made++; *out = x; return 0; }; };
  for (int round = 0; round < 2; round++)
    for (int device = 0; device < 3; device++)
      for (int k = 0; k < 2; k++)
        for (size_t size : {32u, 64u}) {
          const int want = 100 * device + 10 * k + (int)size;
          if (p.find(device, &kernel[k], size, &v, give(want)) || v != want) return 1;
        }
  if (made != 12) return 2;  // once per (device, kernel, size), not once per process
  // a failure is returned and not kept
  if (p.find(5, kernel, 1, &v, [](int *) { return 7; }) != 7) return 3;
  if (p.find(5, kernel, 1, &v, give(4)) || v != 4) return 4;
  // threads that make the first call together
  std::atomic<int> calls{0}, wrong{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 16; t++)
    ts.emplace_back([&, t] {
      for (int i = 0; i < 1000; i++) {
        int x = 0;
        if (p.find(10 + i % 8, kernel, 2, &x, [&, i](int *o) { calls++; *o = i % 8 + 1; return 0; }) || x != i % 8 + 1) wrong++;
      }
    });
  for (auto &t : ts) t.join();
  return wrong ? 5 : calls == 8 ? 0 : 6;
}
"""


def test_found_once_per_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(_PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0


def test_no_kernel_setting_is_kept_per_process():
    """Shared-memory limits are raised by kernel_blocks_per_sm (per device) or for every launch, never behind a static."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        lines = open(os.path.join(CSRC, f)).read().split("\n")
        for i, line in enumerate(lines):
            if "cudaFuncSetAttribute" in line:
                near = "\n".join(lines[max(0, i - 6):i + 1])
                assert "static bool" not in near and "static int" not in near and "static const cudaError_t" not in near, (f, i + 1)

"""What a kernel was configured with belongs to a device: a process that uses a
second one must configure it there too, or launches with more than the default
shared memory fail. The table is host code and runs here with device numbers of
its own; that every attribute goes through it is read from the source."""
import glob
import os
import re
import subprocess

from paper_2110_01011_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.cuh"
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
  rqlp::PerDevice<int> t;
  int v = 0, calls = 0;
  for (int round = 0; round < 3; ++round)
    for (int dev : {0, 1, 63}) {
      CHECK(t.get(dev, &v, [&](int* x) { ++calls; *x = 10 + dev; return 0; }) == 0);
      CHECK(v == 10 + dev);
    }
  CHECK(calls == 3);   // once per device
  // a failure is returned, leaves the other devices alone, and is tried again
  CHECK(t.get(2, &v, [](int*) { return 7; }) == 7);
  CHECK(t.get(1, &v, [](int*) { return 8; }) == 0 && v == 11);
  CHECK(t.get(2, &v, [](int* x) { *x = 5; return 0; }) == 0 && v == 5);
  // beyond the table: asked every time
  for (int i = 0; i < 2; ++i) CHECK(t.get(64, &v, [&](int* x) { ++calls; *x = 1; return 0; }) == 0);
  CHECK(calls == 5);
  // several threads: once, and all of them see it
  rqlp::PerDevice<int> u;
  std::atomic<int> made{0}, wrong{0};
  std::vector<std::thread> th;
  for (int i = 0; i < 8; ++i)
    th.emplace_back([&] {
      for (int dev = 0; dev < 64; ++dev) {
        int x = 0;
        if (u.get(dev, &x, [&](int* y) { ++made; *y = dev + 1; return 0; }) != 0 || x != dev + 1) ++wrong;
      }
    });
  for (auto& h : th) h.join();
  CHECK(made == 64 && wrong == 0);
  return 0;
}
"""


def test_once_per_device_and_again_after_a_failure(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", build.CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_attribute_is_set_once_per_process():
    """cudaFuncSetAttribute and the occupancy queries appear only inside a
    PerDevice's make function."""
    seen = 0
    for f in sorted(glob.glob(os.path.join(build.CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(f).read())
        for m in re.finditer(r"cudaFuncSetAttribute\(|cudaOccupancyMax\w+\(", text):
            before = text[:m.start()]
            at = max(before.rfind("get(current_device()"), 0)
            assert at > 0 and "\n}\n" not in before[at:], (os.path.basename(f), m.group(0))
            seen += 1
        assert not re.search(r"static (bool|int|size_t) \w+ = (false|0);", text), os.path.basename(f)
    assert seen >= 5

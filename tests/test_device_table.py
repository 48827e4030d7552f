"""Per-device values of the launchers (csrc/ff_device.h), compiled and run on the host."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2502_06073_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "ff_device.h"

static std::atomic<int> made[FF_MAX_DEVICES];
static PerDevice<int> table;

int main() {
  std::atomic<int> wrong{0};
  std::vector<std::thread> threads;
  for (int t = 0; t < 8; ++t)
    threads.emplace_back([&] {
      for (int k = 0; k < 1000; ++k)
        for (int dev : {0, 1, 5, FF_MAX_DEVICES - 1}) {
          const int* v = table.get(dev, [dev](int& x) {
            made[dev].fetch_add(1);
            x = 100 + dev;
            return true;
          });
          if (!v || *v != 100 + dev) wrong.fetch_add(1);
        }
    });
  for (auto& t : threads) t.join();
  for (int dev = 0; dev < FF_MAX_DEVICES; ++dev)
    if (made[dev] != (dev == 0 || dev == 1 || dev == 5 || dev == FF_MAX_DEVICES - 1)) wrong++;
  // out of range; a failure is not kept
  auto seven = [](int& x) { x = 7; return true; };
  if (table.get(-1, seven) || table.get(FF_MAX_DEVICES, seven)) wrong++;
  if (table.get(2, [](int&) { return false; })) wrong++;
  const int* v = table.get(2, seven);
  if (!v || *v != 7) wrong++;
  std::printf("%d\n", wrong.load());
  return 0;
}
"""


def test_one_value_per_device_and_thread_safe(tmp_path):
    """Each device's value is made once, whatever the number of threads, and independently of the
    other devices'."""
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-pthread", "-I", CSRC,
                    str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True, timeout=60)
    assert out.stdout.strip() == "0"


def test_no_launcher_keeps_a_device_fact_in_a_plain_static():
    """A static number or flag inside a launcher holds what the first device said for all."""
    for name in os.listdir(CSRC):
        if name.endswith((".cu", ".cuh")):
            text = open(os.path.join(CSRC, name)).read()
            found = re.findall(r"^\s+static (?:int|bool|size_t|long long)\s+\w+\s*=.*$", text, re.M)
            assert not found, (name, found)

"""Kernel attributes and device queries are per CUDA device, not per process."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2505_23429_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
int main() {
  a2::PerDevice<int> v;
  int calls[3] = {0, 0, 0};
  bool threw = false;
  try {
    v.at(2, [&]() -> int { ++calls[2]; throw 1; });
  } catch (int) { threw = true; }
  std::vector<std::thread> t;
  for (int i = 0; i < 8; ++i)
    t.emplace_back([&] { for (int d = 0; d < 3; ++d) v.at(d, [&] { ++calls[d]; return 10 * d + 1; }); });
  for (auto& x : t) x.join();
  int got[3];
  for (int d = 0; d < 3; ++d) got[d] = v.at(d, [] { return -1; });
  bool range = false;
  try { v.at(64, [] { return 0; }); } catch (const std::runtime_error&) { range = true; }
  printf("%d %d %d %d %d %d %d %d\n", calls[0], calls[1], calls[2], got[0], got[1], got[2], threw, range);
}
"""


def test_once_for_every_device(tmp_path):
    src = tmp_path / "t.cc"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["1", "1", "2", "1", "11", "21", "1", "1"]   # a failed first use is repeated


def test_no_attribute_is_set_once_per_process():
    """Attributes are set inside a PerDevice initialiser, or by the call that launches."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"std::call_once\(\w+, \[[^\]]*\] \{(.*?)\n  \}\);", text, re.S):
            for word in ("cudaFuncSetAttribute", "set_smem", "cudaDeviceGetAttribute",
                         "cudaOccupancy"):
                assert word not in m.group(1), (name, m.group(0))

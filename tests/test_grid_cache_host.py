"""Persistent grid sizes are kept per kernel and device (host code; compiled and run here)."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1306_1122_gb300", "csrc")
MAIN = r"""
#include "grid_cache.h"
#include <thread>
int main() {
  dbie::GridCache c;
  int f = 0, g = 0;
  if (c.find(&f, 0) != 0) return 1;
  c.put(&f, 0, 304);
  if (c.find(&f, 0) != 304 || c.find(&f, 1) != 0 || c.find(&g, 0) != 0) return 2;
  c.put(&f, 1, 20);
  c.put(&g, 0, 7);
  c.put(&f, 0, 5);   // the first entry stands
  if (c.find(&f, 0) != 304 || c.find(&f, 1) != 20 || c.find(&g, 0) != 7 || c.find(&g, 1) != 0) return 3;
  std::thread t[4];
  for (int i = 0; i < 4; ++i)
    t[i] = std::thread([&c, i, &f] { for (int d = 2; d < 200; ++d) { c.put(&f, d, d + 1); c.find(&f, i); } });
  for (auto& x : t) x.join();
  for (int d = 2; d < 200; ++d) if (c.find(&f, d) != d + 1) return 4;
  return 0;
}
"""


def test_entries_belong_to_a_device(tmp_path):
    src, exe = tmp_path / "m.cpp", tmp_path / "m"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-pthread", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0

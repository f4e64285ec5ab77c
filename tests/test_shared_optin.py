"""The bookkeeping of shared-memory opt-ins (csrc/bmg_optin.h), compiled for
the host with a fake of the device attribute: asked for on every device of the
process, never lowered, a refusal reported and asked for again."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1803_02481_gb300", "csrc")

PROGRAM = r"""
#include "bmg_optin.h"
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
  bmg::SharedOptIn s;
  int calls = 0, k1 = 0, k2 = 0;
  auto yes = [&](size_t) { ++calls; return true; };
  // every kernel on every device
  for (int round = 0; round < 3; ++round)
    for (int dev = 0; dev < 2; ++dev) {
      CHECK(s.ensure(&k1, dev, 60000, yes));
      CHECK(s.ensure(&k2, dev, 60000, yes));
    }
  CHECK(calls == 4);
  // a smaller size does not ask again, a larger one does
  CHECK(s.ensure(&k1, 0, 50000, yes) && calls == 4);
  CHECK(s.ensure(&k1, 0, 70000, yes) && calls == 5);
  CHECK(s.ensure(&k1, 0, 60000, yes) && calls == 5);
  // a refusal is reported, and not remembered as a grant
  CHECK(!s.ensure(&k1, 1, 90000, [](size_t) { return false; }));
  CHECK(s.ensure(&k1, 1, 60000, yes) && calls == 5);
  CHECK(s.ensure(&k1, 1, 90000, yes) && calls == 6);
  // threads of different sizes: the attribute is never below what a thread was granted
  std::atomic<size_t> attribute{0};
  std::atomic<int> refused{0};
  int k3 = 0;
  std::vector<std::thread> threads;
  for (int t = 0; t < 4; ++t)
    threads.emplace_back([&, t] {
      for (int r = 0; r < 2000; ++r) {
        const size_t bytes = 50000 + 1000 * ((r * 7 + t * 13) % 40);
        s.ensure(&k3, 0, bytes, [&](size_t b) { attribute = b; return true; });
        std::this_thread::yield();
        if (attribute < bytes) ++refused;
      }
    });
  for (auto& t : threads) t.join();
  CHECK(refused == 0);
  return 0;
}
"""


def test_opt_in_bookkeeping(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "optin.cpp", tmp_path / "optin"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout

"""The opt-in to more shared memory than 48 KB holds for one device: it is made on each device that a process
uses, before any caller goes on, and again after a failure. Compiled and run on the host."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_37772_gb300", "csrc")
SRC = r"""
#include "once_per_device.h"
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#define EXPECT(c) if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; }
int main() {
  uad::OncePerDevice once;
  std::vector<int> seen;
  const auto note = [&](int d, int rc) { return once.run(d, [&] { seen.push_back(d); return rc; }); };
  EXPECT(note(0, 0) == 0 && note(0, 0) == 0 && note(1, 0) == 0 && note(0, 0) == 0 && note(1, 0) == 0);
  EXPECT((seen == std::vector<int>{0, 1}));
  EXPECT(note(2, -5) == -5 && note(2, 0) == 0 && note(2, -5) == 0);   // a failure is reported and tried again
  EXPECT(seen.size() == 4);
  std::atomic<int> ready{0}, early{0}, runs{0};
  std::vector<std::thread> ts;
  for (int i = 0; i < 8; ++i)
    ts.emplace_back([&] {
      once.run(7, [&] {
        ++runs;
        std::this_thread::sleep_for(std::chrono::milliseconds(50));
        ready = 1;
        return 0;
      });
      if (!ready) ++early;   // nobody goes on before it is done
    });
  for (auto& t : ts) t.join();
  EXPECT(runs == 1 && early == 0);
  return 0;
}
"""


def test_once_per_device(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    (tmp_path / "t.cc").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-pthread", "-I", CSRC, "-o", str(tmp_path / "t"), str(tmp_path / "t.cc")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_the_projection_kernels_opt_in_once_per_device():
    """No process-wide flag decides whether the projection kernels have been prepared."""
    with open(os.path.join(CSRC, "gemm_tc.cu")) as f:
        src = f.read()
    body = src[src.index("gemm_tc_prepare() {"):]
    body = body[:body.index("\n}\n")]
    assert "OncePerDevice" in body and "static bool" not in body

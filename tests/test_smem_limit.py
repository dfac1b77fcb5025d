"""A kernel's dynamic shared-memory limit is raised and never lowered: on the CPU, against a fake runtime.

`csrc/smem_limit.h` is host code. The fake keeps one limit per kernel, as the runtime does per device. A
launch that was allowed its bytes must still be allowed them after another thread asked for fewer; an
error of either call comes back and sets nothing; and threads that ask for different sizes, each checking
the limit when it would launch, are never refused."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2601_14414_gb300", "csrc")

HARNESS = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "smem_limit.h"
using namespace pimpc;
std::atomic<std::size_t> limit{49152};
struct Fake {
  int get_rc = 0, set_rc = 0;
  int get(std::size_t *b) const { *b = limit; return get_rc; }
  int set(std::size_t b) const { if (set_rc == 0) limit = b; return set_rc; }
};
int main() {
  std::mutex mu;
  const int a = raise_smem_limit(Fake{}, mu, 61488), b = raise_smem_limit(Fake{}, mu, 12000);
  std::printf("%d %d %zu\n", a, b, limit.load());
  const int c = raise_smem_limit(Fake{3, 0}, mu, 90000), d = raise_smem_limit(Fake{0, 5}, mu, 90000);
  std::printf("%d %d %zu\n", c, d, limit.load());
  std::atomic<int> refused{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 4; ++t)
    ts.emplace_back([&, t] {
      for (int i = 0; i < 20000; ++i) {
        const std::size_t want = 61488 + 16 * ((i * 7 + t * 13) % 4096);
        if (raise_smem_limit(Fake{}, mu, want) != 0 || limit < want) ++refused;
      }
    });
  for (auto &t : ts) t.join();
  std::printf("refused %d\n", refused.load());
  return 0;
}
"""


def test_the_limit_is_never_lowered(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()
    assert out == ["0 0 61488", "3 5 61488", "refused 0"]


def test_every_launch_goes_through_it():
    # the only place that sets the attribute is the raising one
    names = [f for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh", ".h"))]
    using = [f for f in names if "cudaFuncAttributeMaxDynamicSharedMemorySize" in open(os.path.join(CSRC, f)).read()]
    assert using == ["misc.cu"]

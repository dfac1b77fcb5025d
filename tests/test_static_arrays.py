"""The momentum table of the no-allocation entry point, on the CPU against a fake runtime.

`csrc/static_arrays.h` is host code: a small program compiled here with g++ gives it a runtime whose
copies reach the device's array only when they are waited for, as a copy from pageable memory may. The
addresses must not be published before the table is there, nor after an error at any of the calls, and
a second call must not touch the runtime again. The factors are compared with the recurrence in
extended precision."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2601_14414_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "static_arrays.h"
using namespace pimpc;
constexpr int kLen = 4096;
struct Fake {
  char scratch_[16];
  double device[kLen] = {};
  std::vector<double> staged;
  int calls = 0, fail_at = 0;
  int step() { return ++calls == fail_at ? 7 : 0; }
  int scratch(void **p) { *p = scratch_; return step(); }
  int table(double **p) { *p = device; return step(); }
  int copy(double *dst, const double *src, int n) {
    const int rc = step();
    if (rc == 0) staged.assign(src, src + n);
    return rc;
  }
  int wait() {
    const int rc = step();
    if (rc == 0) for (size_t i = 0; i < staged.size(); ++i) device[i] = staged[i];
    return rc;
  }
};
int main() {
  for (int fail = 1; fail <= 4; ++fail) {
    Fake f;
    f.fail_at = fail;
    StaticArrays a;
    const int rc = ensure_static_arrays(f, a, kLen);
    std::printf("fail %d rc %d published %d\n", fail, rc, a.scratch || a.coefs ? 1 : 0);
  }
  Fake f;
  StaticArrays a;
  const int rc = ensure_static_arrays(f, a, kLen), first = f.calls;
  const int again = ensure_static_arrays(f, a, kLen);
  std::printf("ok %d %d calls %d %d addresses %d\n", rc, again, first, f.calls,
              a.scratch == f.scratch_ && a.coefs == f.device ? 1 : 0);
  for (int i = 0; i < kLen; ++i) std::printf("%.17g\n", f.device[i]);
  return 0;
}
"""


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("static_arrays")
    src, exe = d / "h.cpp", d / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()


def test_an_error_publishes_nothing(lines):
    assert lines[:4] == [f"fail {i} rc 7 published 0" for i in (1, 2, 3, 4)]


def test_the_table_is_on_the_device_when_the_addresses_are_published(lines):
    assert lines[4] == "ok 0 0 calls 4 4 addresses 1"
    got = np.array([float(v) for v in lines[5:]])
    al, want = np.longdouble(1), []
    for _ in range(len(got)):
        an = (1 + np.sqrt(1 + 4 * al * al)) / 2
        want.append((al - 1) / an)
        al = an
    assert len(got) == 4096 and got[0] == 0.0
    # u = 2^-53: the roundings of m steps leave alpha_m with a relative error of about m u / 2, of which
    # the factor 1 - 1.5 / alpha takes 1.5 / alpha = 3 / m; its own difference and quotient add 2 u
    assert np.max(np.abs(got - np.array(want, np.float64))) <= 8 * 2.0 ** -53

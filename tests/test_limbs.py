"""The integer sum of a warp's floats (csrc/limbs.cuh, host-callable) against exact rational arithmetic:
every lane may lose less than 2^-53 of the largest value's leading bit, what a double addition may
round off, and nothing when the values lie within 2^30 of each other. Spreads up to and beyond that,
subnormals, zeros, all lanes at the largest significand (the limbs' sums must fit 32 bits)."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2601_14414_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <cstdint>
#include "limbs.cuh"
using namespace pimpc::detsum;
int main() {
  unsigned b[32];
  for (;;) {
    for (int i = 0; i < 32; ++i)
      if (std::scanf("%x", &b[i]) != 1) return 0;
    int em = 1;
    for (unsigned v : b) em = (int)(v >> 23) > em ? (int)(v >> 23) : em;
    std::uint64_t lo = 0, hi = 0;
    for (unsigned v : b) {
      const int x = (int)(v >> 23);
      const Limbs q = split((v & 0x7fffffu) | (x ? 0x800000u : 0u), em - (x ? x : 1));
      lo += q.lo;
      hi += q.hi;
    }
    std::printf("%d %llu %d\n", lo >> 32 || hi >> 32 ? 1 : 0, join((unsigned)lo, (unsigned)hi), exponent(em));
  }
}
"""


def cases():
    rng = np.random.default_rng(4)
    out = [np.full(32, np.float32(np.finfo(np.float32).max)), np.zeros(32, np.float32),
           np.full(32, np.nextafter(np.float32(2), np.float32(0)))]
    for spread in (0, 5, 29, 30, 45, 60, 100):
        for at in (-140, -126, -30, 0, 90, 127 - 1):
            for _ in range(4):
                e = np.clip(at - rng.integers(0, spread + 1, 32), -149, 127)
                v = np.ldexp(1.0 + rng.random(32), e).astype(np.float32)
                v[rng.random(32) < 0.1] = 0.0
                out.append(np.minimum(v, np.finfo(np.float32).max))
    return out


def test_sums_lose_less_than_double_additions(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    vals = cases()
    text = "\n".join(" ".join(f"{b:x}" for b in v.view(np.uint32)) for v in vals)
    out = subprocess.run([str(exe)], input=text, check=True, capture_output=True, text=True).stdout.splitlines()
    assert len(out) == len(vals)
    for v, line in zip(vals, out):
        over, sig, e = (int(w) for w in line.split())
        got = Fraction(sig) * Fraction(2) ** e
        want = sum((Fraction(float(x)) for x in v), Fraction(0))
        lead = int(np.frexp(max(float(v.max()), 2.0 ** -126))[1]) - 1  # 2^lead <= the largest value
        lost = want - got
        assert over == 0 and 0 <= lost < 32 * Fraction(2) ** (lead - 53)
        some = v[v > 0]
        if len(some) and np.frexp(float(some.min()))[1] - 1 >= lead - 30:
            assert lost == 0

"""Bringing fixed-point values to a common exponent (fx::scale2 of csrc/fx64.cuh), compiled for the
host and compared with long double: every shift a pass can ask for, on values up to the largest
modulus a stage leaves (2^62.8).  A right shift rounds to nearest, ties to even, so it is off by at
most half a unit whatever the shift; a left shift is exact.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_08578_gb300", "csrc")

# what the headers need of CUDA on the host
HOST = r"""
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdio>
#include <random>
#define __device__
#define __host__
#define __forceinline__ inline
#define __CUDACC__ 1
static struct { int x; } threadIdx;
static inline unsigned __reduce_or_sync(unsigned, unsigned a) { return a; }
static inline void atomicOr(int* p, int v) { *p |= v; }
static inline int __clz(int v) { return v ? __builtin_clz(v) : 32; }
static inline long long __double_as_longlong(double d) { long long r; __builtin_memcpy(&r, &d, 8); return r; }
static inline int __float2int_rz(float f) { return (int)f; }
#include "fft_reg.cuh"
using namespace kss;
typedef long double ld;
typedef std::complex<ld> cld;
"""

SCALES = HOST + r"""
int main() {
  std::mt19937_64 g(1);
  const long long top = (long long)powl(2, 62.8L);
  int bad = 0, odd = 0;
  for (int it = 0; it < 400000; ++it) {
    const int s = (int)(g() % 81) - 10;
    // all sizes and the ends of the range; a left shift only of what it can hold
    long long a = (long long)(g() >> (1 + g() % 63)) % (top + 1);
    if (it % 5 == 0) a = top - (long long)(g() % 1000);
    if (it % 7 == 0 && s > 0 && s < 63) a = (2 * (long long)(g() % 3) + 1) << (s - 1) > top ? a : (2 * (a & 1) + 1) << (s - 1);
    if (s < 0) a >>= -s;
    if (g() & 1) a = -a;
    const ld x = ldexpl((ld)a, -s);
    const long long r = fx::scale2(a, s);
    if (fabsl(x - (ld)r) > 0.5L) ++bad;
    if (fabsl(x - (ld)r) == 0.5L && (r & 1)) ++odd;
  }
  printf("%d %d\n", bad, odd);
}
"""


def run(tmp_path, source):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "t.cpp"
    src.write_text(source)
    subprocess.run([gxx, "-O1", "-std=c++17", "-w", "-I", CSRC, str(src), "-o", str(tmp_path / "t")], check=True)
    return subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True).stdout.split()


def test_shifts_round_to_nearest(tmp_path):
    bad, odd = run(tmp_path, SCALES)
    assert int(bad) == 0   # off by more than half a unit
    assert int(odd) == 0   # a tie that did not go to even

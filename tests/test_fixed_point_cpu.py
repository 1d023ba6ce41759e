"""The fixed-point arithmetic of the double-precision transforms (csrc/fx64.cuh, csrc/fft_reg.cuh),
compiled for the host and compared with long double.

* Every DFT codelet on components up to its stage limit, the corners among them, in both
  directions: an error of a few units, so nothing overflows and no product is lost.
* Rotations at the largest modulus they accept, with low limbs of -2^31 among the inputs.
* Multiplications by V, conversion from double, shifts with ties.

Bounds: a codelet of n points rounds at most three times on the way to an output (n <= 16: two
levels and a factor), each rounding off by at most 3/4 of a unit, summed over at most n terms in
the worst case: 12 units is above what any of them can collect at these sizes; a rotation is off
by at most 1.25 units a component from its two sums, 2.5 in modulus with its factor's error.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_08578_gb300", "csrc")

SRC = r"""
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
static inline int __reduce_max_sync(unsigned, int a) { return a; }
static inline void atomicOr(int* p, int v) { *p |= v; }
static inline void atomicMax(int* p, int v) { *p = std::max(*p, v); }
static inline int __vimax3_s32(int a, int b, int c) { return std::max(a, std::max(b, c)); }
static inline int __vimin3_s32(int a, int b, int c) { return std::min(a, std::min(b, c)); }
static inline int __clz(int v) { return v ? __builtin_clz(v) : 32; }
static inline long long __double_as_longlong(double d) { long long r; __builtin_memcpy(&r, &d, 8); return r; }
static inline int __float2int_rz(float f) { return (int)f; }
#include "fft_reg.cuh"
using namespace kss;
typedef long double ld;
typedef std::complex<ld> cld;
static const ld PI = 3.141592653589793238462643383279502884L;
static cld val(fx::Cx v) { return cld((ld)v.x, (ld)v.y); }
template <int N> ld codelet(int s) {
  std::mt19937_64 g(N);
  ld err = 0;
  const int b = fx::kLimit(N);
  for (int it = 0; it < 1000; ++it) {
    fx::Cx v[N];
    cld in[N];
    for (int i = 0; i < N; ++i) {
      v[i].x = (long long)(g() >> (63 - b)) - (1LL << b);
      v[i].y = (long long)(g() >> (63 - b)) - (1LL << b);
      if (it < 4) {
        v[i].x = it & 1 ? 1LL << b : -(1LL << b);
        v[i].y = it & 2 ? v[i].x : -v[i].x;
      }
      in[i] = val(v[i]);
    }
    fftr::rdft<N>(v, s);
    for (int q = 0; q < N; ++q) {
      cld r = 0;
      for (int t = 0; t < N; ++t) r += in[t] * std::polar((ld)1, s * 2 * PI * ((t * q) % N) / N);
      err = std::max(err, std::abs(r - val(v[q])));
    }
  }
  return err;
}
int main() {
  std::mt19937_64 g(1);
  auto uni = [&] { return (ld)(g() >> 11) * 0x1p-53L; };
  ld c = 0;
  for (int s = -1; s <= 1; s += 2)
    c = std::max({c, codelet<2>(s), codelet<3>(s), codelet<4>(s), codelet<5>(s), codelet<6>(s), codelet<8>(s),
                  codelet<9>(s), codelet<10>(s), codelet<12>(s), codelet<15>(s), codelet<16>(s)});
  ld r = 0;
  for (int it = 0; it < 200000; ++it) {
    const int n = 2 + g() % 255, m = g() % n;
    const cld a = std::polar(powl(2, 62.8L) * (it % 4 ? uni() : 1), 2 * PI * uni());
    fx::Cx v{(long long)a.real(), (long long)a.imag()};
    if (it % 7 == 0) v.x = (v.x & ~0xffffffffLL) | 0x80000000LL;
    if (it % 11 == 0) v.y = (v.y & ~0xffffffffLL) | 0x80000000LL;
    const fx::Rot w = fx::rot_limbs(fx::kcos62(m, n), -fx::ksin62(m, n));
    const cld W = std::polar((ld)1, -2 * PI * m / n);
    r = std::max({r, std::abs(val(v) * W / (ld)4 - val(fx::rot_small<false>(v, w))),
                  std::abs(val(v) * std::conj(W) / (ld)4 - val(fx::rot_small<true>(v, w)))});
  }
  ld p = 0, d = 0, h = 0;
  for (int it = 0; it < 200000; ++it) {
    const long long a = (long long)g() >> 2, f = (long long)((uni() - 0.5L) * 0x1.fffffep63L);
    p = std::max(p, fabsl((ld)a * (ld)f / 0x1p64L - (ld)fx::mulc(a, fx::limbs(f))));
    const double x = ldexp((double)uni() - 0.5, (int)(g() % 80) - 60);
    d = std::max(d, fabsl(ldexpl((ld)x, 41) - (ld)fx::from_double(x, -41)));
    const int s = 1 + g() % 20;
    h = std::max(h, fabsl(ldexpl((ld)(a >> 2), -s) - (ld)fx::shr_round(a >> 2, s)));
    h = std::max(h, fabsl((ld)(a >> 2) / 2 - (ld)fx::half(a >> 2)));
  }
  ld bias = 0;  // ties go to even: no constant is added
  for (long long a = -1000; a < 1000; ++a) bias += (ld)fx::half(a) - (ld)a / 2 + (ld)fx::shr_round(a, 2) - (ld)a / 4;
  printf("%.3Lf %.3Lf %.3Lf %.3Lf %.3Lf %.3Lf\n", c, r, p, d, h, fabsl(bias));
}
"""


def test_fixed_point_arithmetic(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "t.cpp"
    src.write_text(SRC)
    subprocess.run([gxx, "-O1", "-std=c++17", "-w", "-I", CSRC, str(src), "-o", str(tmp_path / "t")], check=True)
    out = subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True).stdout
    codelet, rotation, product, convert, shift, bias = map(float, out.split())
    assert codelet < 12
    assert rotation < 2.5
    assert product < 1.0
    assert convert <= 0.5
    assert shift <= 0.5
    assert bias < 2.0

// Fixed-point arithmetic of the double-precision local passes: complex numbers of two 64-bit
// integers with a power-of-two scale kept per plane of data (block floating point).
//
// Why integers: the FP64 pipe issues 2 lane-operations a clock and SM, the integer pipes 128 adds
// and about 28 32 x 32 + 64-bit multiply-adds, so a 64-bit add costs 1/32 of a DADD and a full
// complex rotation (12 multiply-adds) about a quarter of its four FP64 operations.  A transform
// is additions and rotations of numbers of like size, which is what fixed point does well.
//
// Accuracy: a block whose largest component lies just below 2^b keeps b bits below that
// component; double precision keeps 53 below every single one.  The passes keep b between 54 and
// 62 in every stage, and one rounding costs 0.29 units, so the error of a transform is a few
// 2^-56 of the block's rms (double precision: a few 2^-54; the figures are in local_fx.cuh).
//
// Overflow: a DFT of n points whose component sizes are below 2^b gives outputs of modulus below
// n sqrt(2) 2^b.  Every stage takes its input with b <= kLimit(n), chosen so that the outputs stay
// below 2^62.8, the largest modulus a rotation (rot_*) accepts, whatever the data: the size of a
// stage's input is measured by the stage before it (Mag) and the input shifted right when it is
// too large, and left when it has become small.
#pragma once

#include <cstdint>
#include <type_traits>

namespace kss {
namespace fx {

struct alignas(16) Cx {
  long long x, y;
};
template <typename C> inline constexpr bool is_fx = std::is_same<C, Cx>::value;

// ---- sin and cos of 2 pi m / n in units of 2^-62, from their Taylor series in integers ---------
using i128 = __int128;
constexpr long long kOne62 = 1LL << 62;
__host__ __device__ constexpr long long mul62(long long a, long long b) {
  return (long long)(((i128)a * b + ((i128)1 << 61)) >> 62);
}
// x in [0, pi/4] in units of 2^-62; the terms are formed in units of 2^-62
__host__ __device__ constexpr long long sin62(long long x) {
  const long long x2 = mul62(x, x);
  long long term = x, sum = x;
  for (int k = 1; k < 14 && term != 0; ++k) {
    const long long d = (2LL * k) * (2LL * k + 1);
    term = -((mul62(term, x2) + (term >= 0 ? d / 2 : -d / 2)) / d);
    sum += term;
  }
  return sum;
}
__host__ __device__ constexpr long long cos62(long long x) {
  const long long x2 = mul62(x, x);
  long long term = kOne62, sum = kOne62;
  for (int k = 1; k < 14 && term != 0; ++k) {
    const long long d = (2LL * k - 1) * (2LL * k);
    term = -((mul62(term, x2) + (term >= 0 ? d / 2 : -d / 2)) / d);
    sum += term;
  }
  return sum;
}
// angle (pi/2) r / n for 0 <= 2 r <= n, from pi/2 in units of 2^-62
__host__ __device__ constexpr long long angle62(int r, int n) {
  return (long long)(((i128)7244019458077122842LL * r + n / 2) / n);
}
// cos (q = 0) or sin (q = 1) of (pi/2) r / n, 0 <= r < n
__host__ __device__ constexpr long long quad62(bool s, int r, int n) {
  const bool flip = 2 * r > n;
  const long long a = angle62(flip ? n - r : r, n);
  return s != flip ? sin62(a) : cos62(a);
}
__host__ __device__ constexpr long long kcos62(int m, int n) {
  m %= n;
  if (m < 0) m += n;
  const int q = (4 * m) / n, r = 4 * m - q * n;
  return q == 0 ? quad62(false, r, n) : q == 1 ? -quad62(true, r, n) : q == 2 ? -quad62(false, r, n) : quad62(true, r, n);
}
__host__ __device__ constexpr long long ksin62(int m, int n) {
  m %= n;
  if (m < 0) m += n;
  const int q = (4 * m) / n, r = 4 * m - q * n;
  return q == 0 ? quad62(true, r, n) : q == 1 ? quad62(false, r, n) : q == 2 ? -quad62(true, r, n) : -quad62(false, r, n);
}

// A multiplier as two signed 32-bit limbs, c = h 2^32 + l.
struct Limbs {
  int l, h;
};
__host__ __device__ constexpr Limbs limbs(long long c) {
  return Limbs{(int)(uint32_t)((unsigned long long)c & 0xffffffffull), (int)((c + 0x80000000LL) >> 32)};
}
// One rotation factor (c, s) = (cos, sin) in units of 2^-62, in limbs.
struct alignas(16) Rot {
  int cl, ch, sl, sh;
};
// (c, s) in limbs; a low limb of -2^31 is moved by one unit so that it can be negated
__host__ __device__ constexpr Rot rot_limbs(long long c, long long s) {
  if ((uint32_t)(unsigned long long)c == 0x80000000u) c += 1;
  if ((uint32_t)(unsigned long long)s == 0x80000000u) s += 1;
  const Limbs a = limbs(c), b = limbs(s);
  return Rot{a.l, a.h, b.l, b.h};
}

// Largest b such that a DFT of n points on components below 2^b has outputs of modulus below 2^62.8
__host__ __device__ constexpr int kLimit(int n) {
  int b = 61;
  // (n sqrt(2) 2^b)^2 <= 2^125.6: 2 n^2 <= 2^(125.6 - 2 b), with 2^0.6 >= 1.5
  while (2.0 * n * n > 1.5 * (double)(1ull << (125 - 2 * b > 62 ? 62 : 125 - 2 * b))) --b;
  return b;
}
static_assert(kLimit(4) == 60 && kLimit(8) == 59 && kLimit(12) == 58 && kLimit(16) == 58, "stage limits");

// exponent e with |V| < 2^e (1 - 2^-22), so that V 2^(63 - e) fits two limbs, from the largest high word
__host__ __device__ constexpr int v_exp(int high) {
  const int f = (high + 1) >> 20;
  return (f > 1 ? f : 1) - 1022;
}

// Component i of a slab of size kSlabBits, to time the passes on: the indices hashed, spread evenly over two
// bits less, as in a band most components lie below the largest.  So no stage of the y transform finds its
// input outside its range and stops to shift it (fit).
constexpr int kSlabBits = 59;
__host__ __device__ constexpr long long slab_value(unsigned long long i) {
  unsigned long long h = i * 0x9E3779B97F4A7C15ull + 1;
  h ^= h >> 29;
  h *= 0xBF58476D1CE4E5B9ull;
  return (long long)h >> (65 - kSlabBits);
}

#ifdef __CUDACC__
__device__ __forceinline__ int lo32(long long a) { return (int)a; }
// high limb that goes with the signed low limb
__device__ __forceinline__ int hi_limb(long long a) { return (int)((a + 0x80000000LL) >> 32); }

// round(a c / 2^64) for a constant |c| <= 2^63 (a multiplier of size at most one half), |a| < 2^62.8:
// the product of the low limbs (at most a quarter unit) is left out
__device__ __forceinline__ long long mulc(long long a, Limbs c) {
  const int al = lo32(a), ah = hi_limb(a);
  const long long mid = (long long)ah * c.l + ((long long)al * c.h + 0x80000000LL);
  return (long long)ah * c.h + (mid >> 32);
}
// Shifts round to nearest, ties to even: a tie that always went one way would be a constant added to
// every point of a plane, and a transform collects those of all N^3 points in its G = 0 output
// (measured: 4e-14 of the rms there, 100 times the error of the others).
__device__ __forceinline__ long long half(long long a) { return (a + ((unsigned)a >> 1 & 1u)) >> 1; }
// (a + 2^(s - 1) must be in range)
__device__ __forceinline__ long long shr_round(long long a, int s) {
  return (a + ((1LL << (s - 1)) - 1) + ((a >> s) & 1)) >> s;
}

// a w / 2^64 for the rotation w (or its conjugate), |a| < 2^62.8
template <bool CONJ>
__device__ __forceinline__ Cx rot_small(Cx a, const Rot& w) {
  const int al = lo32(a.x), ah = hi_limb(a.x), bl = lo32(a.y), bh = hi_limb(a.y);
  // w: re = a c - b s, im = a s + b c; conj(w): re = a c + b s, im = b c - a s.  The factor's limbs
  // are negated, not the data's: rot_limbs keeps its low limbs off -2^31
  const int rl = CONJ ? w.sl : -w.sl, rh = CONJ ? w.sh : -w.sh;
  long long m = (long long)ah * w.cl + 0x80000000LL;
  m += (long long)al * w.ch;
  m += (long long)bh * rl;
  m += (long long)bl * rh;
  Cx r;
  r.x = (m >> 32) + (long long)ah * w.ch + (long long)bh * rh;
  long long k = (long long)bh * w.cl + 0x80000000LL;
  k += (long long)bl * w.ch;
  k += (long long)ah * -rl;
  k += (long long)al * -rh;
  r.y = (k >> 32) + (long long)bh * w.ch + (long long)ah * -rh;
  return r;
}

// Size of a block: the OR of the high words' magnitudes of everything a stage stores, gathered in
// a shared word; bits() bounds the components, |v| <= 2^bits.
struct Mag {
  int acc = 0;
  __device__ __forceinline__ void see(long long v) {
    const int h = (int)(v >> 32);
    acc |= h ^ (h >> 31);
  }
  __device__ __forceinline__ void see(Cx v) {
    see(v.x);
    see(v.y);
  }
  // all 32 lanes of every warp call this; the next __syncthreads makes the word complete
  __device__ __forceinline__ void put(int* word) {
    const int w = __reduce_or_sync(0xffffffffu, (unsigned)acc);
    if ((threadIdx.x & 31) == 0 && w) atomicOr(word, w);
  }
};
__device__ __forceinline__ int mag_bits(int word) { return 64 - __clz(word); }
// Shift of a stage's input of size `bits`: right (> 0) to at most `limit`, left (< 0) when it lies
// more than four bits below (then its rms is below 2^52), none for the sizes between.
__device__ __forceinline__ int fit(int bits, int limit) {
  const int d = bits - limit;
  return d > 0 || d < -4 ? d : 0;
}
__device__ __forceinline__ Cx shift(Cx v, int s) {
  if (s > 0) return Cx{shr_round(v.x, s), shr_round(v.y, s)};
  return Cx{v.x << -s, v.y << -s};
}

// a 2^s (s <= 0: left shift by -s, which must not overflow; s > 0: rounded right shift), |a| < 2^62.8.
// shr_round adds half a unit first, which from s = 61 on would leave the range: those shifts round what
// they drop by itself.
__device__ __forceinline__ long long scale2(long long a, int s) {
  if (s <= 0) return a << (s < -63 ? 63 : -s);
  if (s <= 60) return shr_round(a, s);
  if (s > 63) return 0;
  const long long q = a >> s;
  const unsigned long long low = (unsigned long long)a & ((1ULL << s) - 1);
  return q + (long long)((low + ((1ULL << (s - 1)) - 1) + (unsigned long long)(q & 1)) >> s);
}

// A double x = +-m 2^(e - 1075) as an integer multiple of 2^E, rounded; |x| < 2^(E + 63) (finite x)
__device__ __forceinline__ long long from_double(double x, int E) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  long long m = b & 0xfffffffffffffLL;
  if (e) m |= 1LL << 52;
  const int s = (e ? e : 1) - 1075 - E;  // fixed = m 2^s
  if (s >= 0) m <<= s;
  else m = s < -54 ? 0 : (m + (1LL << (-s - 1))) >> -s;
  return b < 0 ? -m : m;
}
#endif

}  // namespace fx
}  // namespace kss

// The passes of the double-precision local part in fixed point (fx64.cuh): the stages, layouts and
// pruning of the CTA-wide passes (local_kernels.cuh) on 64-bit integers with block exponents.
//
//   pass A  one CTA per (z-plane u3, band): the plane's largest component sets its exponent; scatter,
//           inverse x transform, slab plane and its (exponent, size) to fx.ma[band][u3]
//   pass B  one CTA per (x-plane, band): the W3 rows brought to one exponent as they are loaded;
//           y and z transforms, x V, back; (exponent, size) to fx.mb[band][x]
//   pass C  one CTA per (u3, band): the N1 points of a row brought to one exponent; forward x
//           transform, back to double, gather and the Chebyshev epilogue
//
// What bounds them: integer issue.  FP64 runs at 2 lane-operations a clock and SM, which held these
// passes in FP64 at 80 % of that pipe's issue; in integers a butterfly is two 128-lane adds.  Measured
// at the 96-point box, 564 bands (A / B / C, ms): FP64 3.05 / 52.3 / 3.49, fixed point 1.02 / 12.9 /
// 1.41; at the 54-point box, 47 bands (us): 104 / 938 / 111 and 29 / 242 / 39.  Error of T psi + V psi
// against long double, bands falling off as 1 / (1 + T^2), relative to |V psi|: FP64 4.8e-16 and
// fixed point 1.8e-16 at 96 points, 8.2e-16 and 1.8e-16 at 54; flat bands 1.47e-15 and 1.37e-15
// (the rounding of the outputs).
//
// Sizes: a stage of DFT-n takes components below 2^kLimit(n); rotations return their result
// divided by 4, which takes up the growth of the DFTs on either side (about 2^1.7 of the rms each),
// so that a stage's input seldom needs the measured shift.
//
// A non-finite input marks its band (size -1): its outputs are NaN, as the FP64 transform of the
// band would give.
#pragma once

#include "local_kernels.cuh"

namespace kss {
namespace lk {

// Exponents: a value v of a plane with exponent E is v 2^E; size s: all components <= 2^s.
using fx::Cx;
using fx::Rot;

template <int N>
__host__ __device__ constexpr int popcount_mask(unsigned m) {
  int c = 0;
  for (int i = 0; i < N; ++i) c += m >> i & 1u;
  return c;
}

// Brings the n values at p, a stage's input of `bits` bits, to its range; returns the shift.  A
// pass of its own over shared memory, since few stages need it: inside the stages it would double
// their code, which the instruction cache does not hold (measured: 0.95 of a warp's issue slots
// waited for instructions).
__device__ __forceinline__ int refit(Cx* p, int n, int bits, int limit) {
  const int s = fx::fit(bits, limit);
  if (s) {
#pragma unroll 1
    for (int i = threadIdx.x; i < n; i += blockDim.x) p[i] = fx::shift(p[i], s);
    __syncthreads();
  }
  return s;
}

template <int A, int B>
struct FxX {
  static constexpr int N = A * B, P = N + 1;  // the tile index table's pitch
  static size_t smem(int W2) { return sizeof(Rot) * N + sizeof(Cx) * (size_t)W2 * P + sizeof(int) * (4 + N); }
  __device__ static int pos(int x) { return x / A + B * (x % A); }
};

// a.psi of plane u3 and band n as doubles (packed mode: psi_2n + i psi_2n+1 is formed in fixed point)
template <int A, int B, int CW>
__device__ __forceinline__ void fx_pass_a(const LocalArgs<double>& a, int u3, int nl) {
  using G = FxX<A, B>;
  constexpr int N = G::N, P = G::P;
  constexpr unsigned MW = fftr::edge_mask<A, CW>(), MF = fftr::full_mask<A>();
  constexpr int kIn = fx::kLimit(popcount_mask<A>(MW)) - 1;  // one bit for the packed sum
  extern __shared__ __align__(16) unsigned char smraw[];
  Rot* tw = reinterpret_cast<Rot*>(smraw);
  Cx* tile = reinterpret_cast<Cx*>(tw + N);
  int* word = reinterpret_cast<int*>(tile + a.W2 * P);  // exponent field, size after stages 1 and 2
  const int tid = threadIdx.x, NT = blockDim.x;
  const int n = a.n0 + nl;
  int r0 = a.rowrange[2 * u3];
  const int r1 = a.rowrange[2 * u3 + 1];
  const int nrows = r1 >= r0 ? r1 - r0 + 1 : 0;
  if (!nrows) r0 = 0;
  Cx* rows = tile + r0 * P;
  if (tid < 3) word[tid] = 0;
  for (int i = tid; i < N; i += NT) tw[i] = a.fx.r1[i];
  for (int i = tid; i < nrows * P; i += NT) rows[i] = Cx{0, 0};
  const int g0 = a.zstart[u3], g1 = a.zstart[u3 + 1];
  const double2* pa = a.psi + (size_t)(a.packed ? 2 * n : n) * a.ld;
  const double2* pb = a.packed && 2 * n + 1 < a.nbands ? pa + a.ld : nullptr;
  unsigned em = 0;
  auto field = [&](double v) { em = max(em, (unsigned)__double2hiint(v) >> 20 & 0x7ffu); };
  for (int g = g0 + tid; g < g1; g += NT) {
    const double2 x = pa[g];
    field(x.x);
    field(x.y);
    if (pb) {
      const double2 y = pb[g];
      field(y.x);
      field(y.y);
    }
  }
  em = __reduce_max_sync(0xffffffffu, em);
  __syncthreads();
  if ((tid & 31) == 0 && em) atomicMax(word, (int)em);
  __syncthreads();
  const int e = word[0];
  const bool bad = e == 0x7ff;
  const int E = max(e, 1) - 1022 - kIn;  // every |component| < 2^(E + kIn)
  for (int g = g0 + tid; g < g1; g += NT) {
    const double2 x = pa[g];
    Cx v{fx::from_double(x.x, E), fx::from_double(x.y, E)};
    if (pb) {  // x + i y
      const double2 y = pb[g];
      v.x -= fx::from_double(y.y, E);
      v.y += fx::from_double(y.x, E);
    }
    tile[a.tileidx[g]] = v;
  }
  __syncthreads();
  const fftr::FastDiv dnr(nrows > 0 ? nrows : 1);
  // inverse, stage 1
  fx::Mag mag;
  for (int t = tid; t < nrows * B; t += NT) {
    const int r = dnr(t), u = t - r * nrows;
    Cx* row = rows + u * P + r;
    Cx v[A];
    fftr::static_for<0, A>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      if constexpr (MW >> i & 1u) v[i] = row[B * i];
    });
    fftr::rdft_m<A, MW, MF>(v, 1);
    v[0].x = fx::shr_round(v[0].x, 2);
    v[0].y = fx::shr_round(v[0].y, 2);
#pragma unroll
    for (int k = 1; k < A; ++k) v[k] = fx::rot_small<true>(v[k], tw[r * k]);
#pragma unroll
    for (int k = 0; k < A; ++k) {
      mag.see(v[k]);
      row[B * k] = v[k];
    }
  }
  mag.put(word + 1);
  __syncthreads();
  const int sh = refit(rows, nrows * P, fx::mag_bits(word[1]), fx::kLimit(B));
  fx::Mag mag2;
  for (int t = tid; t < nrows * A; t += NT) {
    const int k = dnr(t), u = t - k * nrows;
    Cx* row = rows + u * P + B * k;
    Cx v[B];
#pragma unroll
    for (int j = 0; j < B; ++j) v[j] = row[j];
    fftr::rdft<B>(v, 1);
#pragma unroll
    for (int j = 0; j < B; ++j) {
      mag2.see(v[j]);
      row[j] = v[j];
    }
  }
  mag2.put(word + 2);
  __syncthreads();
  Cx* dst = reinterpret_cast<Cx*>(a.work) + ((size_t)nl * N * a.W3 + u3) * a.W2;
  const size_t xs = (size_t)a.W3 * a.W2;
  const fftr::FastDiv dw2(a.W2);
  for (int i = tid; i < N * a.W2; i += NT) {
    const int x = dw2(i), u2 = i - x * a.W2;
    const int u = u2 - r0;
    dst[x * xs + u2] = (u >= 0 && u < nrows) ? rows[u * P + G::pos(x)] : Cx{0, 0};
  }
  if (tid == 0)
    a.fx.ma[(size_t)nl * a.W3 + u3] = make_int2(E + 2 + sh, bad ? -1 : fx::mag_bits(word[2]));
}

template <int A, int B>
struct FxB {
  static constexpr int N = A * B;
  static constexpr int QS = (N + 1) | 1, ZS = (N + 1) | 1;  // odd pitches, as WideB
  static size_t smem(int W3) {
    return sizeof(Rot) * N + sizeof(Cx) * ((size_t)W3 * QS + (size_t)N * ZS) + sizeof(int) * (N + W3 + 10);
  }
};

// Shared memory of a plane's y and z transforms (pass B, density).
template <int A, int B>
struct FxPlane {
  using G = FxB<A, B>;
  Rot* tw;
  Cx* Q;      // W3 rows (z in the sphere window) x N (y)
  Cx* Z;      // N columns (y position) x N (z)
  int* zmap;
  int* rs;    // shift of each row at the load
  int* word;  // sizes after each of 8 stages, top exponent, bad
  __device__ FxPlane(const LocalArgs<double>& a, unsigned char* sm) {
    tw = reinterpret_cast<Rot*>(sm);
    Q = reinterpret_cast<Cx*>(tw + G::N);
    Z = Q + a.W3 * G::QS;
    zmap = reinterpret_cast<int*>(Z + G::N * G::ZS);
    rs = zmap + G::N;
    word = rs + a.W3;
  }
  // the rotations and the window's z map, once per CTA
  __device__ void tables(const LocalArgs<double>& a) const {
    for (int i = threadIdx.x; i < G::N; i += blockDim.x) tw[i] = a.fx.r2[i];
    for (int z = threadIdx.x; z < G::N; z += blockDim.x) {
      int u = (z - a.lo3) % G::N;
      if (u < 0) u += G::N;
      zmap[z] = u < a.W3 ? u : -1;
    }
  }
};

// Slab plane (x, nl) through the y transform and the first stage of the z transform: Z ready for its
// DFT-B stage (in that stage's range), values v 2^E.  Returns E; bad: the band is not finite.
template <int A, int B, int CW>
__device__ __forceinline__ int fx_inverse(const LocalArgs<double>& a, int x, int nl, const FxPlane<A, B>& s,
                                          bool& bad) {
  using G = FxB<A, B>;
  constexpr int N = G::N, QS = G::QS, ZS = G::ZS;
  constexpr unsigned MW = fftr::edge_mask<A, CW>(), MF = fftr::full_mask<A>();
  constexpr int kWin = fx::kLimit(popcount_mask<A>(MW));
  const Rot* tw = s.tw;
  Cx *Q = s.Q, *Z = s.Z;
  const int* zmap = s.zmap;
  int *rs = s.rs, *word = s.word;
  const int tid = threadIdx.x, NT = blockDim.x;
  const int W3 = a.W3, W2 = a.W2;
  if (tid < 10) word[tid] = tid == 8 ? INT_MIN / 2 : 0;
  for (int i = tid; i < W3 * QS; i += NT) Q[i] = Cx{0, 0};
  const int2* ma = a.fx.ma + (size_t)nl * W3;
  __syncthreads();
  for (int u = tid; u < W3; u += NT) {
    const int2 m = ma[u];
    rs[u] = m.x;
    if (m.y < 0) word[9] = 1;
    else atomicMax(word + 8, m.x + m.y);
  }
  __syncthreads();
  constexpr int kLoad = kWin - 1;  // leaves the shift after the first stage to the exception
  bad = word[9] != 0;
  int E = (word[8] == INT_MIN / 2 ? 0 : word[8]) - kLoad;
  const Cx* slab = reinterpret_cast<const Cx*>(a.work) + ((size_t)nl * a.N1 + x) * W3 * W2;
  const fftr::FastDiv dw2(W2), dw3(W3);
  for (int i = tid; i < W3 * W2; i += NT) {
    const int u3 = dw2(i), u2 = i - u3 * W2;
    const int s = E - rs[u3];
    Cx v = slab[i];
    v.x = fx::scale2(v.x, s);
    v.y = fx::scale2(v.y, s);
    Q[u3 * QS + fftr::wrap_add(a.lo2, u2, N)] = v;
  }
  __syncthreads();
  // ---- y, inverse ----
  {
    fx::Mag mag;
    for (int t = tid; t < W3 * B; t += NT) {
      const int r = dw3(t), u = t - r * W3;
      Cx* row = Q + u * QS + r;
      Cx v[A];
      fftr::static_for<0, A>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        if constexpr (MW >> i & 1u) v[i] = row[B * i];
      });
      fftr::rdft_m<A, MW, MF>(v, 1);
      v[0].x = fx::shr_round(v[0].x, 2);
      v[0].y = fx::shr_round(v[0].y, 2);
#pragma unroll
      for (int k = 1; k < A; ++k) v[k] = fx::rot_small<true>(v[k], tw[r * k]);
#pragma unroll
      for (int k = 0; k < A; ++k) {
        mag.see(v[k]);
        row[B * k] = v[k];
      }
    }
    mag.put(word + 0);
  }
  __syncthreads();
  int sh = refit(Q, W3 * QS, fx::mag_bits(word[0]), fx::kLimit(B));
  E += 2 + sh;
  {
    fx::Mag mag;
    for (int t = tid; t < W3 * A; t += NT) {
      const int k = dw3(t), u = t - k * W3;
      Cx* row = Q + u * QS + B * k;
      Cx v[B];
#pragma unroll
      for (int j = 0; j < B; ++j) v[j] = row[j];
      fftr::rdft<B>(v, 1);
#pragma unroll
      for (int j = 0; j < B; ++j) {
        mag.see(v[j]);
        row[j] = v[j];
      }
    }
    mag.put(word + 1);
  }
  __syncthreads();
  // ---- z, inverse stage 1 ----
  sh = refit(Q, W3 * QS, fx::mag_bits(word[1]), kWin);
  E += 2 + sh;
  {
    fx::Mag mag;
    for (int t = tid; t < N * B; t += NT) {
      const int r = t / N, p = t - r * N;
      Cx v[A];
      fftr::static_for<0, A>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        if constexpr (MW >> i & 1u) {
          const int u = zmap[r + B * i];
          v[i] = u >= 0 ? Q[u * QS + p] : Cx{0, 0};
        }
      });
      fftr::rdft_m<A, MW, MF>(v, 1);
      v[0].x = fx::shr_round(v[0].x, 2);
      v[0].y = fx::shr_round(v[0].y, 2);
#pragma unroll
      for (int k = 1; k < A; ++k) v[k] = fx::rot_small<true>(v[k], tw[r * k]);
      Cx* col = Z + p * ZS + r;
#pragma unroll
      for (int k = 0; k < A; ++k) {
        mag.see(v[k]);
        col[B * k] = v[k];
      }
    }
    mag.put(word + 2);
  }
  __syncthreads();
  sh = refit(Z, N * ZS, fx::mag_bits(word[2]), fx::kLimit(B));
  return E + sh;
}

template <int A, int B, int CW>
__device__ __forceinline__ void fx_pass_b(const LocalArgs<double>& a, int x, int nl) {
  using G = FxB<A, B>;
  constexpr int N = G::N, QS = G::QS, ZS = G::ZS;
  constexpr unsigned MW = fftr::edge_mask<A, CW>(), MF = fftr::full_mask<A>();
  extern __shared__ __align__(16) unsigned char smraw[];
  const FxPlane<A, B> pl(a, smraw);
  const Rot* tw = pl.tw;
  Cx *Q = pl.Q, *Z = pl.Z;
  const int* zmap = pl.zmap;
  int* word = pl.word;
  const int tid = threadIdx.x, NT = blockDim.x;
  const int W3 = a.W3, W2 = a.W2;
  const fftr::FastDiv dw2(W2), dw3(W3);
  pl.tables(a);
  bool bad;
  int E = fx_inverse<A, B, CW>(a, x, nl, pl, bad) + 1;  // V / 2
  int sh;
  // ---- z, inverse stage 2, x V / 2 ----
  {
    fx::Mag mag;
    const fx::Limbs* vp = a.fx.V + (size_t)x * N * N;
    for (int t = tid; t < N * A; t += NT) {
      const int k = t / N, p = t - k * N;
      const fx::Limbs* vrow = vp + (size_t)k * N + p;  // (z = k + A k2, p) at vrow[A k2 N]
      Cx* col = Z + p * ZS + B * k;
      Cx v[B];
#pragma unroll
      for (int j = 0; j < B; ++j) v[j] = col[j];
      fftr::rdft<B>(v, 1);
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) {
        const fx::Limbs vv = vrow[(size_t)A * k2 * N];
        v[k2].x = fx::mulc(v[k2].x, vv);
        v[k2].y = fx::mulc(v[k2].y, vv);
        mag.see(v[k2]);
        col[k2] = v[k2];
      }
    }
    mag.put(word + 3);
  }
  __syncthreads();
  // ---- z, forward stage 1 (its own loop, so that its input is measured: V takes 2^3 to 2^4 off the
  // rms, and a bound over both transforms another 2^4) ----
  {
    const int bits = fx::mag_bits(word[3]);
    sh = refit(Z, N * ZS, max(bits, fx::kLimit(B)), fx::kLimit(B));
    const int up = max(fx::kLimit(B) - bits, 0);  // left shift, as the values are loaded
    E += 2 + sh - up;
    fx::Mag mag;
    for (int t = tid; t < N * A; t += NT) {
      const int k = t / N, p = t - k * N;
      Cx* col = Z + p * ZS + B * k;
      Cx v[B];
#pragma unroll
      for (int j = 0; j < B; ++j) v[j] = Cx{col[j].x << up, col[j].y << up};
      fftr::rdft<B>(v, -1);
      v[0].x = fx::shr_round(v[0].x, 2);
      v[0].y = fx::shr_round(v[0].y, 2);
#pragma unroll
      for (int q = 1; q < B; ++q) v[q] = fx::rot_small<false>(v[q], tw[k * q]);
#pragma unroll
      for (int q = 0; q < B; ++q) {
        mag.see(v[q]);
        col[q] = v[q];
      }
    }
    mag.put(word + 4);
  }
  __syncthreads();
  // ---- z, forward stage 2: keep the window rows ----
  sh = refit(Z, N * ZS, fx::mag_bits(word[4]), fx::kLimit(A));
  E += sh;
  {
    fx::Mag mag;
    for (int t = tid; t < N * B; t += NT) {
      const int q = t / N, p = t - q * N;
      const Cx* col = Z + p * ZS + q;
      Cx v[A];
#pragma unroll
      for (int m = 0; m < A; ++m) v[m] = col[B * m];
      fftr::rdft_m<A, MF, MW>(v, -1);
      fftr::static_for<0, A>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        if constexpr (MW >> k & 1u) {
          const int u = zmap[q + B * k];
          if (u >= 0) {
            mag.see(v[k]);
            Q[u * QS + p] = v[k];
          }
        }
      });
    }
    mag.put(word + 5);
  }
  __syncthreads();
  // ---- y, forward ----
  sh = refit(Q, W3 * QS, fx::mag_bits(word[5]), fx::kLimit(B));
  E += 2 + sh;
  {
    fx::Mag mag;
    for (int t = tid; t < W3 * A; t += NT) {
      const int r = dw3(t), u = t - r * W3;
      Cx* row = Q + u * QS + B * r;
      Cx v[B];
#pragma unroll
      for (int j = 0; j < B; ++j) v[j] = row[j];
      fftr::rdft<B>(v, -1);
      v[0].x = fx::shr_round(v[0].x, 2);
      v[0].y = fx::shr_round(v[0].y, 2);
#pragma unroll
      for (int q = 1; q < B; ++q) v[q] = fx::rot_small<false>(v[q], tw[r * q]);
#pragma unroll
      for (int q = 0; q < B; ++q) {
        mag.see(v[q]);
        row[q] = v[q];
      }
    }
    mag.put(word + 6);
  }
  __syncthreads();
  sh = refit(Q, W3 * QS, fx::mag_bits(word[6]), fx::kLimit(A));
  E += sh;
  {
    fx::Mag mag;
    for (int t = tid; t < W3 * B; t += NT) {
      const int q = dw3(t), u = t - q * W3;
      Cx* row = Q + u * QS + q;
      Cx v[A];
#pragma unroll
      for (int m = 0; m < A; ++m) v[m] = row[B * m];
      fftr::rdft_m<A, MF, MW>(v, -1);
      fftr::static_for<0, A>([&](auto kc) {  // rows outside the window are not read again
        constexpr int k = decltype(kc)::value;
        if constexpr (MW >> k & 1u) {
          mag.see(v[k]);
          row[B * k] = v[k];
        }
      });
    }
    mag.put(word + 7);
  }
  __syncthreads();
  Cx* slab = reinterpret_cast<Cx*>(a.work) + ((size_t)nl * a.N1 + x) * W3 * W2;
  for (int i = tid; i < W3 * W2; i += NT) {
    const int u3 = dw2(i), u2 = i - u3 * W2;
    slab[i] = Q[u3 * QS + fftr::wrap_add(a.lo2, u2, N)];
  }
  if (tid == 0) a.fx.mb[(size_t)nl * a.N1 + x] = make_int2(E, bad ? -1 : fx::mag_bits(word[7]));
}

template <int A, int B, int CW>
__device__ __forceinline__ void fx_pass_c(const LocalArgs<double>& a, int u3, int nl) {
  using G = FxX<A, B>;
  constexpr int N = G::N, P = G::P;
  constexpr unsigned MW = fftr::edge_mask<A, CW>(), MF = fftr::full_mask<A>();
  constexpr int kIn = fx::kLimit(B);
  extern __shared__ __align__(16) unsigned char smraw[];
  Rot* tw = reinterpret_cast<Rot*>(smraw);
  Cx* tile = reinterpret_cast<Cx*>(tw + N);
  int* word = reinterpret_cast<int*>(tile + a.W2 * P);  // top exponent, bad, size after stage 1
  int* xs_e = word + 4;                                 // exponent of each x-plane
  const int tid = threadIdx.x, NT = blockDim.x;
  const int n = a.n0 + nl;
  int r0 = a.rowrange[2 * u3];
  const int r1 = a.rowrange[2 * u3 + 1];
  const int nrows = r1 >= r0 ? r1 - r0 + 1 : 0;
  if (!nrows) r0 = 0;
  Cx* rows = tile + r0 * P;
  if (tid < 3) word[tid] = tid == 0 ? INT_MIN / 2 : 0;
  for (int i = tid; i < N; i += NT) tw[i] = a.fx.r1[i];
  __syncthreads();
  const int2* mb = a.fx.mb + (size_t)nl * N;
  for (int x = tid; x < N; x += NT) {
    const int2 m = mb[x];
    xs_e[x] = m.x;
    if (m.y < 0) word[1] = 1;
    else atomicMax(word, m.x + m.y);
  }
  __syncthreads();
  const bool bad = word[1] != 0;
  int E = (word[0] == INT_MIN / 2 ? 0 : word[0]) - kIn;
  const Cx* src = reinterpret_cast<const Cx*>(a.work) + ((size_t)nl * N * a.W3 + u3) * a.W2;
  const size_t xs = (size_t)a.W3 * a.W2;
  const fftr::FastDiv dnr(nrows > 0 ? nrows : 1);
  for (int i = tid; i < N * nrows; i += NT) {
    const int x = dnr(i), u = i - x * nrows;
    const int s = E - xs_e[x];
    Cx v = src[x * xs + r0 + u];
    v.x = fx::scale2(v.x, s);
    v.y = fx::scale2(v.y, s);
    rows[u * P + G::pos(x)] = v;
  }
  __syncthreads();
  {
    fx::Mag mag;
    for (int t = tid; t < nrows * A; t += NT) {
      const int r = dnr(t), u = t - r * nrows;
      Cx* row = rows + u * P + B * r;
      Cx v[B];
#pragma unroll
      for (int j = 0; j < B; ++j) v[j] = row[j];
      fftr::rdft<B>(v, -1);
      v[0].x = fx::shr_round(v[0].x, 2);
      v[0].y = fx::shr_round(v[0].y, 2);
#pragma unroll
      for (int q = 1; q < B; ++q) v[q] = fx::rot_small<false>(v[q], tw[r * q]);
#pragma unroll
      for (int q = 0; q < B; ++q) {
        mag.see(v[q]);
        row[q] = v[q];
      }
    }
    mag.put(word + 2);
  }
  __syncthreads();
  const int sh = refit(rows, nrows * P, fx::mag_bits(word[2]), fx::kLimit(A));
  E += 2 + sh;
  for (int t = tid; t < nrows * B; t += NT) {
    const int q = dnr(t), u = t - q * nrows;
    Cx* row = rows + u * P + q;
    Cx v[A];
#pragma unroll
    for (int m = 0; m < A; ++m) v[m] = row[B * m];
    fftr::rdft_m<A, MF, MW>(v, -1);
    fftr::static_for<0, A>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      if constexpr (MW >> k & 1u) row[B * k] = v[k];
    });
  }
  __syncthreads();
  // back to double: v 2^E / (N1 N2 N3), in two factors when the first alone would leave the normal range
  E += fx::v_exp(*a.fx.vhigh);
  const bool tiny = E < -900;
  const double sc = bad ? __longlong_as_double(0x7ff8000000000000LL) : ldexp(a.fx.invn, tiny ? E + 600 : E);
  const double sc2 = tiny ? 0x1p-600 : 1.0;
  auto val = [&](long long v) {
    const double d = (double)v * sc;
    return tiny ? d * sc2 : d;
  };
  const int g0 = a.zstart[u3], g1 = a.zstart[u3 + 1];
  double2* po = a.out + n * a.ld;
  if (a.packed) {
    for (int g = g0 + tid; g < g1; g += NT) {
      const Cx v = tile[a.tileidx[g]];
      po[g] = make_double2(val(v.x), val(v.y));
    }
    return;
  }
  const double2* ps = a.psi + n * a.ld;
  const double2* pp = a.psi_prev ? a.psi_prev + n * a.ld : nullptr;
  const double al = a.coef ? a.coef[0] : a.alpha;
  const double be = a.coef ? a.coef[1] : a.beta;
  const double ga = a.coef ? a.coef[2] : a.gamma;
  for (int g = g0 + tid; g < g1; g += NT) {
    const Cx v = tile[a.tileidx[g]];
    const double2 p = ps[g];
    const double t = a.kin[g];
    double2 o;
    o.x = al * (t * p.x + val(v.x)) + be * p.x;
    o.y = al * (t * p.y + val(v.y)) + be * p.y;
    if (pp) {
      const double2 q = pp[g];
      o.x += ga * q.x;
      o.y += ga * q.y;
    }
    po[g] = o;
  }
}

}  // namespace lk
}  // namespace kss

// Density of double-precision bands on the fixed-point transforms (local_fx.cuh): per (x-plane, band
// group) the inverse y and z transforms of each band's plane and the accumulation of w |psi|^2.
//
// What bounds it: integer issue (the transforms), with the FP64 pipe beside it: |psi|^2 is formed
// from 32-bit limbs as a 64-bit integer in units of 2^62 (four multiply-adds instead of two FP64
// operations at 1/14 of their rate; its rounding is below 2^-60 of it), and only its
// conversion and the weighted sum (3 FP64 operations a point) are left on that pipe.
//
// Measured, 96-point box, 512 bands: 8.8 ms (FP64: 32), pass A 0.95.  Sum over the box against the
// bands' norms: off by 2e-17 (24, 54 and 96 points; FP64, whose rounded twiddles act on every band alike:
// 2.4e-16 to 8.2e-16).
#include "density.h"
#include "local_fx_impl.cuh"

namespace kss {

namespace {

using namespace lk;
using fx_detail::edge;
using fx_detail::kFxThreads;

// (x^2 + y^2) / 2^62 of |v| < 2^62.8, zero for zero.  The squares of the low limbs (each at most one
// unit, two thirds together on average) are left out; rounding the middle product up adds one half
__device__ __forceinline__ unsigned long long norm62(Cx v) {
  const int al = fx::lo32(v.x), ah = fx::hi_limb(v.x), bl = fx::lo32(v.y), bh = fx::hi_limb(v.y);
  const long long hi = (long long)ah * ah + (long long)bh * bh;
  const long long mid = (long long)ah * al + ((long long)bh * bl + 0x1fffffffLL);
  return (unsigned long long)((hi << 2) + (mid >> 29));
}

template <int A, int B, int CW>
__global__ void __launch_bounds__(kFxThreads) pass_df(LocalArgs<double> a, int m, int G, const double* __restrict__ occ,
                                                      double* __restrict__ part) {
  pdl_wait();
  using W = FxB<A, B>;
  constexpr int N = W::N, ZS = W::ZS, NT = kFxThreads;
  constexpr int R = (N * A + NT - 1) / NT;
  extern __shared__ __align__(16) unsigned char smraw[];
  const FxPlane<A, B> pl(a, smraw);
  const int x = blockIdx.x, g = blockIdx.y, tid = threadIdx.x;
  pl.tables(a);
  double acc[R][B];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int j = 0; j < B; ++j) acc[r][j] = 0;
#pragma unroll 1
  for (int b = g; b < m; b += G) {
    __syncthreads();  // the previous band's reads are done
    bool bad;
    const int E = fx_inverse<A, B, CW>(a, x, b, pl, bad);
    // |psi|^2 = norm62 2^(2 E + 62).  norm62 becomes a double through the high and low words in the
    // fraction fields of 2^84 and 2^52 (2^84 + 2^52 subtracted), whose exponents also take the scale as
    // far as it fits; the rest goes to the weight.
    const int k = 2 * E + 62, kf = min(max(k, -900), 900);
    const double wb = bad ? __longlong_as_double(0x7ff8000000000000LL) : ldexp(occ[a.n0 + b], k - kf);
    const int mh = 0x45300000 + (kf << 20), ml = 0x43300000 + (kf << 20);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int t = tid + NT * r;
      if (t < N * A) {
        const int q = t / N, p = t - q * N;  // columns fastest across lanes
        const Cx* col = pl.Z + p * ZS + B * q;
        Cx v[B];
#pragma unroll
        for (int j = 0; j < B; ++j) v[j] = col[j];
        fftr::rdft<B>(v, 1);
#pragma unroll
        for (int j = 0; j < B; ++j) {
          // the point brought to the top of its range: sizes within a plane differ by 2^10 and more
          const int hx = (int)(v[j].x >> 32), hy = (int)(v[j].y >> 32);
          const int sh = max(__clz((hx ^ (hx >> 31)) | (hy ^ (hy >> 31))) - 2, 0);
          const unsigned long long u = norm62(Cx{v[j].x << sh, v[j].y << sh});
          const int de = sh << 21;  // 2^(-2 sh)
          const double d = (__hiloint2double(mh - de, (int)(u >> 32)) - __hiloint2double(mh - de, 0x00100000)) +
                           __hiloint2double(ml - de, (int)u);
          acc[r][j] = fma(wb, d, acc[r][j]);
        }
      }
    }
  }
  // To the partial plane in natural y, z order, through shared memory (as pass_dw).
  __syncthreads();
  double* st = reinterpret_cast<double*>(pl.Z);
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int t = tid + NT * r;
    if (t < N * A) {
      const int q = t / N, p = t - q * N;
#pragma unroll
      for (int j = 0; j < B; ++j) st[p * ZS + q + A * j] = acc[r][j];
    }
  }
  __syncthreads();
  double* pg = part + ((size_t)g * a.N1 + x) * N * N;
  for (int i = tid; i < N * N; i += NT) {
    const int y = i / N, z = i - y * N;
    const int k2 = y / A, q = y - k2 * A;  // y = q + A k2 sits at position k2 + B q
    pg[i] += st[(k2 + B * q) * ZS + z];
  }
}

template <int A, int B>
bool launch_df(const LocalArgs<double>& a, int m, int G, const double* occ, double* part, cudaStream_t st,
               int* resident) {
  const size_t sm = FxB<A, B>::smem(a.W3);
  if (sm > kWideSmemMax) return false;
  constexpr int PC = edge(A);
  const int cw = wide_prune_cw(A, B, a.lo2, a.W2, a.lo3, a.W3);
  const auto k = PC > 0 && cw > 0 && cw <= PC ? pass_df<A, B, PC> : pass_df<A, B, 0>;
  KSS_CHECK_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  if (resident)
    KSS_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(resident, k, kFxThreads, sm));
  else
    launch_pdl(k, dim3(a.N1, G), kFxThreads, sm, st, a, m, G, occ, part);
  return true;
}

}  // namespace

bool density_pass_fx(const LocalArgs<double>& a, int A, int B, int m, int G, const double* occ, double* part,
                     cudaStream_t st, int* resident) {
  if (a.N2 != a.N3 || A * B != a.N2) return false;
  switch (A * 32 + B) {
#define KSS_CASE(x, y) \
  case x * 32 + y:     \
    return launch_df<x, y>(a, m, G, occ, part, st, resident);
    KSS_SPLITS(KSS_CASE)
#undef KSS_CASE
    default:
      return false;
  }
}

}  // namespace kss

// Kernel instances of the CTA-wide passes (local_kernels.cuh) for one precision: pass B
// (pass_bw_body) for every split of KSS_WIDE_SPLITS, run at 256 or 384 threads per CTA (and 128 in
// single precision), passes A and C (pass_aw_body, pass_cw_body) for the x splits of
// KSS_WIDEX_SPLITS.  Included by one translation unit per precision (local_wide_f32.cu,
// local_wide_f64.cu).  Double precision takes them where the fixed-point passes (local_fx_impl.cuh)
// have no instance: an x edge outside KSS_FX_X, or N2 != N3 with a CTA-wide x edge.
#pragma once

#include "local_kernels.cuh"
#include "local_wide.h"
#include "pdl.cuh"

namespace kss {
namespace wide_detail {

using namespace lk;

template <typename T, int A, int B, int CW>
__global__ void __launch_bounds__(kWideThreads) pass_bw(LocalArgs<T> a) {
  pdl_wait();
  pass_bw_body<T, A, B, CW>(a, blockIdx.x, blockIdx.y);
}

// Every split has two instances: the full transform, and the one pruned to the window that a box of the
// default size leaves (wide_edge).
template <typename T, int A, int B>
bool launch_one(const LocalArgs<T>& a, int nt, int nbands, cudaStream_t st, bool dry) {
  const size_t sm = WideB<T, A, B>::smem(a.W3);
  if (sm > kWideSmemMax) return false;
  if (dry) return true;
  constexpr int PC = wide_edge(A);
  const int cw = wide_prune_cw(A, B, a.lo2, a.W2, a.lo3, a.W3);
  const auto k = PC > 0 && cw > 0 && cw <= PC ? pass_bw<T, A, B, PC> : pass_bw<T, A, B, 0>;
  allow_smem(k, sm);
  launch_pdl(k, dim3(a.N1, nbands), nt, sm, st, a);
  return true;
}

// 128 threads: for the small boxes of batched systems a stage's tasks fill a 128-thread CTA better,
// and four-warp barriers idle fewer warps.
template <typename T>
bool dispatch(const LocalArgs<T>& a, int A, int B, int nt, int nbands, cudaStream_t st, bool dry) {
  if (a.N2 != a.N3 || A * B != a.N2 || (nt != 256 && nt != 384 && (nt != 128 || sizeof(T) == 8))) return false;
  switch (A * 32 + B) {
#define KSS_CASE(x, y) \
  case x * 32 + y:     \
    return launch_one<T, x, y>(a, nt, nbands, st, dry);
    KSS_WIDE_SPLITS(KSS_CASE)
#undef KSS_CASE
    default:
      return false;
  }
}

// ---- passes A and C ----
// x splits with CTA-wide instances (N1 = A * B even) for pass A and for pass C, each with a full form and
// one pruned to the window that a box of the default size leaves (wide_edge).  Each pass puts the
// stage with the twiddle multiply on the 8-point transforms (pass A inverts 8 x 12, pass C forwards
// 12 x 8).  The slab between the passes is in natural x order, so the two passes need not share a
// split.  Shorter edges stay with the per-warp codelets (45 points, 82 bands: 13.9 and 14.3 us per
// warp, 14.4 and 14.3 CTA-wide).
#define KSS_WIDEX_SPLITS(X) X(8, 12, 12, 8)
constexpr int kWideXThreads = 256;

template <typename T, int A, int B, int NT, int CW = 0>
__global__ void __launch_bounds__(NT) pass_aw(LocalArgs<T> a) {
  pdl_wait();
  pass_aw_body<T, A, B, NT, CW>(a, blockIdx.x, blockIdx.y);
}
template <typename T, int A, int B, int NT, int CW = 0>
__global__ void __launch_bounds__(NT) pass_cw(LocalArgs<T> a) {
  pdl_wait();
  pass_cw_body<T, A, B, NT, CW>(a, blockIdx.x, blockIdx.y);
}

template <typename T, int NT, class K>
void launch_x1(K kern, const LocalArgs<T>& a, size_t sm, int nbands, cudaStream_t st) {
  allow_smem(kern, sm);
  launch_pdl(kern, dim3(a.W3, nbands), NT, sm, st, a);
}

// which = 0: pass A (inverse transforms), 1: pass C (forward transforms)
template <typename T, int A, int B, int NT, int which>
bool launch_x(const LocalArgs<T>& a, int nbands, cudaStream_t st, bool dry) {
  using G = WideX<T, A, B>;
  if (a.N1p != G::P) return false;  // the tile index table's pitch
  const size_t sm = G::smem(a.W2);
  if (sm > kWideSmemMax) return false;
  if (dry) return true;
  constexpr int PC = wide_edge(A);
  const bool pruned = PC > 0 && axis_prune_cw(B, a.lo1, a.W1) <= PC;
  if constexpr (which == 0) {
    if (pruned) launch_x1<T, NT>(pass_aw<T, A, B, NT, PC>, a, sm, nbands, st);
    else launch_x1<T, NT>(pass_aw<T, A, B, NT>, a, sm, nbands, st);
  } else {
    if (pruned) launch_x1<T, NT>(pass_cw<T, A, B, NT, PC>, a, sm, nbands, st);
    else launch_x1<T, NT>(pass_cw<T, A, B, NT>, a, sm, nbands, st);
  }
  return true;
}

template <typename T>
bool dispatch_x(const LocalArgs<T>& a, int which, int nbands, cudaStream_t st, bool dry) {
  switch (a.N1) {
#define KSS_CASE(xa, ya, xc, yc)                                                           \
  case xa * ya:                                                                            \
    static_assert(xa * ya == xc * yc, "passes A and C split the same length");            \
    return which == 0 ? launch_x<T, xa, ya, kWideXThreads, 0>(a, nbands, st, dry)          \
                      : launch_x<T, xc, yc, kWideXThreads, 1>(a, nbands, st, dry);
    KSS_WIDEX_SPLITS(KSS_CASE)
#undef KSS_CASE
    default:
      return false;
  }
}

}  // namespace wide_detail
}  // namespace kss

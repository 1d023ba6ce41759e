// Kernel instances of the fixed-point passes (local_fx.cuh).  Pass B: every split of
// KSS_WIDE_SPLITS, run at 256 or 384 threads per CTA; passes A and C: one split for each length of
// KSS_FX_X.  Each has two instances: the full transform, and the one pruned to the window that a
// box of the default size leaves (N >= 4 max|m| + 1, so |m| < N / 4: the first and last
// ceil(A / 4) of a strided stage's A positions).  The instances are spread over several
// translation units, which compile in parallel.
#pragma once

#include "local_fx.cuh"
#include "local_wide.h"
#include "pdl.cuh"

namespace kss {
namespace fx_detail {

using namespace lk;

constexpr int kFxThreads = 384;   // the most a pass-B launch uses (its register allocation)
constexpr int kFxXThreads = 256;

// edge width of the pruned instance of a DFT-A stage, 0 when there is nothing to prune
constexpr int edge(int A) { return 2 * ((A + 3) / 4) < A ? (A + 3) / 4 : 0; }
constexpr int part_of(int A, int B) { return (A * 3 + B) % 4; }

template <int A, int B, int CW>
__global__ void __launch_bounds__(kFxThreads) pass_bf(LocalArgs<double> a) {
  pdl_wait();
  fx_pass_b<A, B, CW>(a, blockIdx.x, blockIdx.y);
}
template <int A, int B, int CW>
__global__ void __launch_bounds__(kFxXThreads) pass_af(LocalArgs<double> a) {
  pdl_wait();
  fx_pass_a<A, B, CW>(a, blockIdx.x, blockIdx.y);
}
template <int A, int B, int CW>
__global__ void __launch_bounds__(kFxXThreads) pass_cf(LocalArgs<double> a) {
  pdl_wait();
  fx_pass_c<A, B, CW>(a, blockIdx.x, blockIdx.y);
}

using Kern = void (*)(LocalArgs<double>);
inline void launch(Kern k, const LocalArgs<double>& a, int gx, int nbands, int nt, size_t sm, cudaStream_t st) {
  allow_smem(k, sm);
  // put in place early only up to about a wave of CTAs (H on 20 bands of 24 planes: 59.6 -> 54.3 us; filter
  // step of 564 bands of 96 planes: 18.37 -> 18.80 ms, the next pass taking places from this one's tail)
  launch_pdl_if((long long)gx * nbands <= 1024, k, dim3(gx, nbands), nt, sm, st, a);
}

template <int PART>
bool dispatch_b(const LocalArgs<double>& a, int A, int B, int nt, int nbands, cudaStream_t st, bool dry);
bool dispatch_a(const LocalArgs<double>& a, int nbands, cudaStream_t st, bool dry);
bool dispatch_c(const LocalArgs<double>& a, int nbands, cudaStream_t st, bool dry);

template <int PART, int A, int B>
bool launch_b(const LocalArgs<double>& a, int nt, int nbands, cudaStream_t st, bool dry) {
  if constexpr (part_of(A, B) == PART) {
    const size_t sm = FxB<A, B>::smem(a.W3);
    if (sm > kWideSmemMax) return false;
    if (dry) return true;
    constexpr int PC = edge(A);
    const int cw = wide_prune_cw(A, B, a.lo2, a.W2, a.lo3, a.W3);
    launch(PC > 0 && cw > 0 && cw <= PC ? (Kern)pass_bf<A, B, PC> : (Kern)pass_bf<A, B, 0>, a, a.N1, nbands, nt, sm, st);
    return true;
  } else {
    return false;
  }
}

// Lengths with fixed-point x passes, N1 = A * B: pass A inverts A x B and pass C forwards B x A's
// mirror, so that the rotations sit on the shorter DFT in both.
#define KSS_FX_X(X) X(3, 5) X(4, 4) X(3, 6) X(4, 5) X(4, 6) X(5, 5) X(3, 9) X(5, 6) X(6, 6) X(5, 8) X(5, 9) \
                    X(6, 8) X(5, 10) X(6, 9) X(6, 10) X(8, 12)

}  // namespace fx_detail
}  // namespace kss

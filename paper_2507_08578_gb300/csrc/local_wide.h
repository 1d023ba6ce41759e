// Host entries of the CTA-wide passes (local_wide_impl.cuh) and of their fixed-point form in double
// precision (local_fx_impl.cuh).
#pragma once

#include "local_kernels.cuh"

namespace kss {

constexpr size_t kWideSmemMax = 227 * 1024;

// Launches pass B for nbands bands (grid N1 x nbands, nt = 256 or 384 threads per CTA) with the
// CTA-wide transform stages for the split N2 == N3 == A * B.  Returns false (and launches
// nothing) when no instance exists for (A, B, nt) or its shared memory does not fit.
// dry = true only checks availability.
template <typename T>
bool wide_pass_b(const lk::LocalArgs<T>& a, int A, int B, int nt, int nbands, cudaStream_t st, bool dry);

// Launches pass A (which = 0) or pass C (which = 1) for nbands bands (grid W3 x nbands) with the
// CTA-wide x transforms (lk::pass_aw_body, lk::pass_cw_body), pruned to the sphere's x window when
// an instance covers it.  Returns false (and launches nothing) when no instance exists for N1 or
// its shared memory does not fit; dry = true only checks availability.
template <typename T>
bool wide_pass_x(const lk::LocalArgs<T>& a, int which, int nbands, cudaStream_t st, bool dry);

// The same in fixed point: pass B (256 or 384 threads), passes A and C.
bool fx_pass_b(const lk::LocalArgs<double>& a, int A, int B, int nt, int nbands, cudaStream_t st, bool dry);
bool fx_pass_x(const lk::LocalArgs<double>& a, int which, int nbands, cudaStream_t st, bool dry);

// Whether all three passes of `a` have a fixed-point instance (the slab between them is in that form, so
// it is all or none): the x edge, and one split of N2 == N3 at least.
bool fx_available(const lk::LocalArgs<double>& a);
template <typename T>
bool fx_available_t(const lk::LocalArgs<T>& a) {
  if constexpr (sizeof(T) == 8) return fx_available(a);
  else return false;
}

// The (A, B) pairs with instances, in KSS_WIDE_SPLITS order.
inline const std::vector<std::pair<int, int>>& wide_splits() {
  static const std::vector<std::pair<int, int>> v = {
#define KSS_PAIR(x, y) {x, y},
      KSS_WIDE_SPLITS(KSS_PAIR)
#undef KSS_PAIR
  };
  return v;
}

}  // namespace kss

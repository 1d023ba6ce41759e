// Double precision of the CTA-wide passes: the fixed-point kernels (local_fx_impl.cuh).
#include "local_fx_impl.cuh"

namespace kss {

template <>
bool wide_pass_b<double>(const lk::LocalArgs<double>& a, int A, int B, int nt, int nbands, cudaStream_t st,
                         bool dry) {
  if (a.N2 != a.N3 || A * B != a.N2 || (nt != 256 && nt != 384)) return false;
  switch (fx_detail::part_of(A, B)) {
    case 0: return fx_detail::dispatch_b<0>(a, A, B, nt, nbands, st, dry);
    case 1: return fx_detail::dispatch_b<1>(a, A, B, nt, nbands, st, dry);
    case 2: return fx_detail::dispatch_b<2>(a, A, B, nt, nbands, st, dry);
    default: return fx_detail::dispatch_b<3>(a, A, B, nt, nbands, st, dry);
  }
}

template <>
bool wide_pass_x<double>(const lk::LocalArgs<double>& a, int which, int nbands, cudaStream_t st, bool dry) {
  return which == 0 ? fx_detail::dispatch_a(a, nbands, st, dry) : fx_detail::dispatch_c(a, nbands, st, dry);
}

}  // namespace kss

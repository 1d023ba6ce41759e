// Host entries of the fixed-point passes (instances: local_fx_impl.cuh and the files that include it).
#include "local_fx_impl.cuh"

namespace kss {

bool fx_pass_b(const lk::LocalArgs<double>& a, int A, int B, int nt, int nbands, cudaStream_t st, bool dry) {
  if (a.N2 != a.N3 || A * B != a.N2 || (nt != 256 && nt != 384)) return false;
  switch (fx_detail::part_of(A, B)) {
    case 0: return fx_detail::dispatch_b<0>(a, A, B, nt, nbands, st, dry);
    case 1: return fx_detail::dispatch_b<1>(a, A, B, nt, nbands, st, dry);
    case 2: return fx_detail::dispatch_b<2>(a, A, B, nt, nbands, st, dry);
    default: return fx_detail::dispatch_b<3>(a, A, B, nt, nbands, st, dry);
  }
}

bool fx_pass_x(const lk::LocalArgs<double>& a, int which, int nbands, cudaStream_t st, bool dry) {
  return which == 0 ? fx_detail::dispatch_a(a, nbands, st, dry) : fx_detail::dispatch_c(a, nbands, st, dry);
}

bool fx_available(const lk::LocalArgs<double>& a) {
  if (a.N2 != a.N3 || !fx_pass_x(a, 0, 0, nullptr, true) || !fx_pass_x(a, 1, 0, nullptr, true)) return false;
  for (const auto& ab : wide_splits())
    if (ab.first * ab.second == a.N2 && fx_pass_b(a, ab.first, ab.second, lk::kWideThreads, 0, nullptr, true)) return true;
  return false;
}

}  // namespace kss

// Fixed-point pass B, part 3 of the splits (local_fx_impl.cuh).
#include "local_fx_impl.cuh"

namespace kss {
namespace fx_detail {

template <>
bool dispatch_b<3>(const LocalArgs<double>& a, int A, int B, int nt, int nbands, cudaStream_t st, bool dry) {
  switch (A * 32 + B) {
#define KSS_CASE(x, y) \
  case x * 32 + y:     \
    return launch_b<3, x, y>(a, nt, nbands, st, dry);
    KSS_WIDE_SPLITS(KSS_CASE)
#undef KSS_CASE
    default:
      return false;
  }
}

}  // namespace fx_detail
}  // namespace kss

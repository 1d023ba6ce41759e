// Fixed-point pass A (scatter and inverse x transform), see local_fx_impl.cuh.
#include "local_fx_impl.cuh"

namespace kss {
namespace fx_detail {

namespace {
template <int A, int B>
bool launch_x(const LocalArgs<double>& a, int nbands, cudaStream_t st, bool dry) {
  using G = FxX<A, B>;
  if (a.N1p != G::P) return false;  // the tile index table's pitch
  const size_t sm = G::smem(a.W2);
  if (sm > kWideSmemMax) return false;
  if (dry) return true;
  constexpr int PC = edge(A);
  const bool pruned = PC > 0 && axis_prune_cw(B, a.lo1, a.W1) <= PC;
  launch(pruned ? (Kern)pass_af<A, B, PC> : (Kern)pass_af<A, B, 0>, a, a.W3, nbands, kFxXThreads, sm, st);
  return true;
}
}  // namespace

bool dispatch_a(const LocalArgs<double>& a, int nbands, cudaStream_t st, bool dry) {
  switch (a.N1) {
#define KSS_CASE(x, y) \
  case x * y:          \
    return launch_x<x, y>(a, nbands, st, dry);
    KSS_FX_X(KSS_CASE)
#undef KSS_CASE
    default:
      return false;
  }
}

}  // namespace fx_detail
}  // namespace kss

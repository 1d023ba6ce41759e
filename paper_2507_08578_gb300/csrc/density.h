// Shared by the density build (density.cu) and the local passes (local_apply.cu).
#pragma once

#include <functional>

#include "local_kernels.cuh"

namespace kss {

// Kernel arguments of the local passes for nb bands of psi (band-major, leading dimension ld).
template <typename T>
lk::LocalArgs<T> density_args(kss_sys s, int ik, const void* psi, int ld);

// Pass A (sphere -> slab: scatter and inverse x transform) of the nb bands of `a` (density_args) in
// chunks that keep the slab L2-resident; after(a, m) is called once per chunk with a.work holding the
// slabs of bands a.n0 .. a.n0 + m - 1.  fx: double precision in fixed point (the slab and a.fx.ma as
// the fixed-point pass A leaves them; the caller has checked that it has an instance).
// KSS_ENOTSUP for FFT lengths without a two-codelet split.
template <typename T>
void pass_a_chunks(kss_sys s, int ik, int nb, lk::LocalArgs<T> a, bool fx,
                   const std::function<void(const lk::LocalArgs<T>&, int)>& after);

// The density accumulation on a fixed-point slab (density_fx.cu): m bands in G groups into the
// partial planes.  False when there is no instance for N2 = N3 = A * B or its shared memory does not
// fit; resident (when given) only receives the resident CTAs per SM, and nothing is launched.
bool density_pass_fx(const lk::LocalArgs<double>& a, int A, int B, int m, int G, const double* occ, double* part,
                     cudaStream_t st, int* resident);

}  // namespace kss

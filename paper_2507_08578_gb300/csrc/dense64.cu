// FP64 dense generalised Hermitian eigensolver for the Rayleigh-Ritz step (§5.1: the subspace
// problem of the Chebyshev-filtered iteration, "less efficient on GPU" and called rarely).
//
// Solves A x = lambda B x for Hermitian A and Hermitian positive definite B (n x n, complex128,
// column-major, lower triangles read), returning all eigenvalues ascending and B-orthonormal
// eigenvectors, in five phases written out here:
//
//   1. Cholesky B = L L^H (blocked right-looking: a 16-column panel at a time, its diagonal block
//      factored in shared memory, the rows below solved against it, then a rank-16 update of the
//      trailing lower triangle).
//   2. Reduction to standard form C = L^{-1} A L^{-H}: two forward substitutions with n
//      right-hand sides each (X = L^{-1} A, then C = L^{-1} X^H, using A = A^H).
//   3. Householder tridiagonalisation C = Q T Q^H (unblocked, on the full Hermitian matrix):
//      per column, the reflector H = I - tau v v^H with a real subdiagonal (beta = -sign(Re
//      alpha) |x|), p = tau C v, w = p - (tau/2)(p^H v) v, C <- C - v w^H - w v^H.
//   4. Eigenpairs of the real symmetric tridiagonal T: every eigenvalue by interpolation and
//      sections on the Sturm count (the number of negative pivots of the LDL^T factorisation of T - sigma I),
//      every eigenvector by inverse iteration with the partially pivoted LU of T - lambda I;
//      eigenvalues closer than 1e-5 |T| form a cluster whose vectors are orthogonalised against
//      each other (modified Gram-Schmidt) in every iteration.
//   5. Back-transformation x = L^{-H} Q z (the reflectors applied to each column of Z in
//      reverse order, then a backward substitution with L^H).
//
// Real symmetric pencils (the Gamma point) run the same phases in real arithmetic on compact real
// copies of the lower triangles: a quarter of the FP64 operations of the O(n^3) phases.
//
// Parallel organisation.  The same phase code runs on a "team": one CTA (barrier = __syncthreads) or
// a cluster of up to eight per pencil of a batch (barrier = the cluster's), or a whole cooperative grid
// (one large pencil, barrier = a grid barrier of this file with a bounded wait).  Work that is independent per
// column (the triangular solves, the reflector applications, the inverse iterations) needs no
// team barrier: one warp owns a column, and what its lanes exchange goes by shuffles or behind a
// warp barrier.
// The barrier count is about n + n/8 per pencil (one per tridiagonalisation step, two per 16-column
// Cholesky panel).
//
// Every grid-barrier wait gives up after a time limit; the kernel then raises the control
// block's error word, sets the pencil's info to -1, and every thread leaves at its next barrier;
// callers report KSS_ETIMEOUT.  A non-positive Cholesky pivot at column j stops the solve with
// info = j + 1 (the LAPACK convention) and leaves the outputs undefined.
#include <cuda/atomic>

#include <algorithm>
#include <cmath>
#include <vector>

#include "kss_internal.h"
#include "recip64.cuh"

namespace kss {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
static_assert((kWarps & (kWarps - 1)) == 0, "the CTA reductions take a power-of-two warp count");

__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }

// ---- complex helpers ---------------------------------------------------------------------------
// On GB300 an SM retires about two FP64 fused multiply-adds per clock, so every FP64 instruction
// counts: complex products are written as chains of fused multiply-adds (4 per complex
// multiply-accumulate) and scalars a whole warp or CTA needs are computed once and broadcast.
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cmulc(double2 a, double2 b) {  // conj(a) * b
  return make_double2(fma(a.x, b.x, a.y * b.y), fma(a.x, b.y, -a.y * b.x));
}
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c) {  // c + a b
  return make_double2(fma(-a.y, b.y, fma(a.x, b.x, c.x)), fma(a.y, b.x, fma(a.x, b.y, c.y)));
}
__device__ __forceinline__ double2 cfms(double2 a, double2 b, double2 c) {  // c - a b
  return make_double2(fma(a.y, b.y, fma(-a.x, b.x, c.x)), fma(-a.y, b.x, fma(-a.x, b.y, c.y)));
}
__device__ __forceinline__ double2 cfmac(double2 a, double2 b, double2 c) {  // c + conj(a) b
  return make_double2(fma(a.y, b.y, fma(a.x, b.x, c.x)), fma(-a.y, b.x, fma(a.x, b.y, c.y)));
}
__device__ __forceinline__ double2 conjd(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
__device__ __forceinline__ double2 shfl_c(double2 v, int src) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ double2 warp_sum_c(double2 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
  }
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The same operations on real scalars: the phases are templates on the scalar type S (double2 for
// Hermitian pencils, double for real symmetric ones, which then take a quarter of the FP64 work of
// the O(n^3) phases and half the memory traffic).
__device__ __forceinline__ double cmul(double a, double b) { return a * b; }
__device__ __forceinline__ double cmulc(double a, double b) { return a * b; }
__device__ __forceinline__ double cfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double cfms(double a, double b, double c) { return fma(-a, b, c); }
__device__ __forceinline__ double cfmac(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double conjd(double a) { return a; }
__device__ __forceinline__ double cadd(double a, double b) { return a + b; }
__device__ __forceinline__ double csub(double a, double b) { return a - b; }
__device__ __forceinline__ double cscale(double a, double s) { return a * s; }
__device__ __forceinline__ double shfl_c(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ double warp_sum_c(double v) { return warp_sum(v); }
__device__ __forceinline__ double shfl_xor_c(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double re(double a) { return a; }
__device__ __forceinline__ double re(double2 a) { return a.x; }
__device__ __forceinline__ double im(double) { return 0.0; }
__device__ __forceinline__ double im(double2 a) { return a.y; }
template <class S>
__device__ __forceinline__ S mk(double x, double y);
template <>
__device__ __forceinline__ double mk<double>(double x, double) { return x; }
template <>
__device__ __forceinline__ double2 mk<double2>(double x, double y) { return make_double2(x, y); }
// s + |a|^2
__device__ __forceinline__ double abs2_acc(double a, double s) { return fma(a, a, s); }
__device__ __forceinline__ double abs2_acc(double2 a, double s) { return fma(a.x, a.x, fma(a.y, a.y, s)); }
// 1 / a
__device__ __forceinline__ double cinv(double a) { return fast_rcp(a); }
__device__ __forceinline__ double2 cinv(double2 a) {
  const double r = fast_rcp(fma(a.x, a.x, a.y * a.y));
  return make_double2(a.x * r, -a.y * r);
}
// complex128 value of a scalar (the caller's matrices are complex128 in both cases)
__device__ __forceinline__ double2 widen(double a) { return make_double2(a, 0.0); }
__device__ __forceinline__ double2 widen(double2 a) { return a; }

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Control block of one grid-team solve (zeroed before the launch).
constexpr int kCounters = 8;
struct Ctl {
  unsigned count[kCounters][32];  // barrier arrivals (monotonic), each counter on a line of its own
  int err;  // 1: a barrier wait gave up
  int pad1;
  unsigned long long t[8];  // %globaltimer at the start and after each phase (measurement)
};

struct CtaTeam {
  __device__ int cta() const { return 0; }
  __device__ int ctas() const { return 1; }
  __device__ int rank() const { return threadIdx.x; }
  __device__ int swrank() const { return threadIdx.x >> 5; }  // rank for per-warp work
  __device__ int size() const { return blockDim.x; }
  __device__ int wsize() const { return blockDim.x >> 5; }
  __device__ bool sync() const {
    __syncthreads();
    return true;
  }
  __device__ void stamp(int) const {}
};

// The CTAs of one thread-block cluster: barriers in hardware (all CTAs of a cluster are resident), which
// also order the CTAs' global writes.
struct ClusterTeam {
  int crank, csize;
  __device__ int cta() const { return crank; }
  __device__ int ctas() const { return csize; }
  __device__ int rank() const { return crank * blockDim.x + threadIdx.x; }
  __device__ int swrank() const { return (threadIdx.x >> 5) * csize + crank; }
  __device__ int size() const { return csize * blockDim.x; }
  __device__ int wsize() const { return csize * (blockDim.x >> 5); }
  __device__ bool sync() const {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
    return true;
  }
  __device__ void stamp(int) const {}
};

struct GridTeam {
  Ctl* ctl;
  int* info;  // the pencil's status word: -1 when a barrier wait gave up
  unsigned long long limit_ns;
  __device__ int cta() const { return blockIdx.x; }
  __device__ int ctas() const { return gridDim.x; }
  __device__ int rank() const { return blockIdx.x * blockDim.x + threadIdx.x; }
  // rank for per-warp independent work, spread over the CTAs first so that n work items use every
  // SM's FP64 units instead of the first few CTAs'
  __device__ int swrank() const { return (threadIdx.x >> 5) * gridDim.x + blockIdx.x; }
  __device__ int size() const { return gridDim.x * blockDim.x; }
  __device__ int wsize() const { return (gridDim.x * blockDim.x) >> 5; }
  // time stamp k (by one thread, after the barrier that ends a phase)
  __device__ void stamp(int k) const {
    if (rank() == 0) ctl->t[k] = global_ns();
  }
  // Grid barrier (all CTAs are resident: cooperative launch).  The counters only grow: barrier number b
  // (counted by every thread in its own copy of the team) is passed once every counter holds b arrivals
  // of each of its CTAs (those with its number modulo kCounters: a single counter takes 150 arrivals
  // one after another).  Each CTA arrives with one release add, which makes the writes of all its
  // threads (ordered before it by __syncthreads) visible to any thread that acquires the counter;
  // eight lanes acquire one counter each, in a bounded spin.  Returns false when the solve has been
  // abandoned.
  mutable unsigned epoch = 0;
  __device__ bool sync() const {
    __shared__ int s_ok;
    __syncthreads();
    ++epoch;
    if (threadIdx.x < 32) {
      const int c = threadIdx.x & (kCounters - 1);
      cuda::atomic_ref<unsigned, cuda::thread_scope_device> cnt(ctl->count[c][0]);
      cuda::atomic_ref<int, cuda::thread_scope_device> err(ctl->err);
      const unsigned target = epoch * ((gridDim.x + kCounters - 1 - c) / kCounters);
      int ok = __all_sync(0xffffffffu, err.load(cuda::memory_order_relaxed) == 0);
      if (ok) {
        if (threadIdx.x < kCounters && (blockIdx.x & (kCounters - 1)) == threadIdx.x)
          cnt.fetch_add(1u, cuda::memory_order_release);
        const unsigned long long t0 = global_ns();
        unsigned spins = 0;
        while (!__all_sync(0xffffffffu, threadIdx.x >= kCounters || cnt.load(cuda::memory_order_acquire) >= target)) {
          if ((++spins & 63u) == 0) {
            const bool late = global_ns() - t0 > limit_ns;
            if (__any_sync(0xffffffffu, late || err.load(cuda::memory_order_relaxed))) {
              if (threadIdx.x == 0 && err.exchange(1, cuda::memory_order_relaxed) == 0) *info = -1;
              ok = 0;
              break;
            }
          }
        }
      }
      if (threadIdx.x == 0) s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
  }
};

// One pencil and its workspace.  For a complex pencil (S = double2) A and B are the caller's
// matrices, worked on in place; for a real one (S = double) they are compact real copies (ld n) in
// the workspace, and the results are written back to the caller's complex matrices at the end.
template <class S>
struct Pencil {
  S* A;         // n x n (lda): in A, out eigenvectors
  S* B;         // n x n (ldb): in B, out Cholesky factor L (lower)
  double* w;    // n eigenvalues (out)
  int* info;    // out: 0, or j + 1 for a non-positive pivot at column j
  int n, lda, ldb;
  S* R;         // n x n (ld n): reduction workspace, then the reflector vectors
  double* Z;    // n x n (ld n): eigenvectors of T
  double* wk;   // 6 n^2 doubles: inverse-iteration arrays
  double* vec;  // 11 n + 8 doubles: d, e, tau (S), p (2 x S), 1/L_jj, q (2)
  int smem_cols;  // 1: the launch gives every warp n words of S of dynamic shared memory
  int resident;   // 1: and the tridiagonalisation its CTA's columns (beside its three vectors)
  double2* outA;  // the caller's A and B (complex128; the same as A and B when S = double2)
  double2* outB;
  int ldoa, ldob;
};

// ---- phase 0: inputs ---------------------------------------------------------------------------
// Real pencils: the real parts of the lower triangles into the compact copies.
template <class Team>
__device__ bool prepare(const Team& T, const Pencil<double>& P) {
  const int n = P.n, lane = threadIdx.x & 31;
  for (int c = T.swrank(); c < n; c += T.wsize()) {
    const double2* __restrict__ ia = P.outA + (size_t)c * P.ldoa;
    const double2* __restrict__ ib = P.outB + (size_t)c * P.ldob;
    double* __restrict__ a = P.A + (size_t)c * P.lda;
    double* __restrict__ b = P.B + (size_t)c * P.ldb;
    for (int i = c + lane; i < n; i += 32) {
      a[i] = ia[i].x;
      b[i] = ib[i].x;
    }
  }
  return T.sync();
}
template <class Team>
__device__ bool prepare(const Team&, const Pencil<double2>&) {
  return true;  // worked on in place
}

// Real pencils: L (lower triangle) back into the caller's B.
template <class Team>
__device__ void finish(const Team& T, const Pencil<double>& P) {
  const int n = P.n, lane = threadIdx.x & 31;
  for (int c = T.swrank(); c < n; c += T.wsize()) {
    const double* __restrict__ b = P.B + (size_t)c * P.ldb;
    double2* __restrict__ ob = P.outB + (size_t)c * P.ldob;
    for (int i = c + lane; i < n; i += 32) ob[i] = make_double2(b[i], 0.0);
  }
}
template <class Team>
__device__ void finish(const Team&, const Pencil<double2>&) {}

// ---- phase 1: Cholesky B = L L^H -----------------------------------------------------------------
template <class S>
__device__ __forceinline__ double* vrdiag(const Pencil<S>& P) { return P.vec + 8 * P.n; }

// Panel width of the blocked Cholesky.
constexpr int kPanel = 16;
// Shared memory of the blocked Cholesky: the diagonal block (pitch panel + 1) and its 1 / L[j][j].
template <class S> __host__ __device__ constexpr size_t chol_smem() {
  return sizeof(S) * (size_t)kPanel * (kPanel + 1) + sizeof(double) * kPanel;
}

// Blocked right-looking Cholesky B = L L^H in panels of W columns, two team barriers per panel:
//   1. every CTA factors the W x W diagonal block in its own shared memory (the same arithmetic
//      in every CTA, so the copies agree bit for bit; the team's first CTA writes it back), one
//      entry of the triangle per thread;
//   2. the rows below it are solved against it, L21 = A21 L11^{-H}, four rows a warp: eight groups of
//      lanes hold two columns each and pass every finished column on by shuffles;
//   3. barrier; the trailing lower triangle is updated, A22 -= L21 L21^H, a warp per 32 rows of
//      one column, one row per lane, the column's W factors broadcast once; barrier.
// What bounds it: a warp's FP64 instruction takes 64 cycles of its quarter of the SM, so each step is
// spread until no warp has a long list of them, and the update's tasks are equal (columns of
// the triangle in pairs of constant length).  Cycles per panel (diagonal / rows / update), order 564
// complex: 23k / 11k / 18k (one warp, 32 rows a warp, a warp a column: 53k / 35k / 48k); 1127 real:
// 19k / 5k / 18k (26k / 11k / 33k).
// Returns false when the solve stops (non-positive pivot: *info set; or an abandoned barrier).
template <class Team, class S>
__device__ bool cholesky(const Team& T, const Pencil<S>& P, S* smem) {
  constexpr int W = kPanel, LP = W + 1;
  static_assert(W == 16, "the lane maps below");
  const int n = P.n, ld = P.ldb;
  S* B = P.B;
  double* rd = vrdiag(P);
  S* Lb = smem;  // diagonal block, column-major with pitch LP
  double* rdb = reinterpret_cast<double*>(Lb + W * LP);
  __shared__ int s_bad;
  const int tid = threadIdx.x, lane = tid & 31;
  const bool first_cta = T.rank() < (int)blockDim.x;
  // entry (di, dk), di >= dk, of thread tid < W (W + 1) / 2: columns of the triangle one after another
  int di = tid, dk = 0;
  while (dk < W && di >= W - dk) {
    di -= W - dk;
    ++dk;
  }
  di += dk;
  const bool mine = dk < W;
  const int nwt = (W * (W + 1) / 2 + 31) / 32;  // warps with entries
  for (int p0 = 0; p0 < n; p0 += W) {
    const int w = min(W, n - p0);
    // 1. the diagonal block
    if (tid < W) rdb[tid] = 0.0;
    if (tid == 0) s_bad = 0;
    S c = mk<S>(0.0, 0.0);
    if (mine) {
      if (di < w) c = B[(p0 + di) + (size_t)(p0 + dk) * ld];
      Lb[dk * LP + di] = c;
    }
    __syncthreads();
    for (int j = 0; j < w; ++j) {
      const double d = re(Lb[j * LP + j]);
      const bool bad = !(d > 0.0) || !isfinite(d);
      if (bad && tid == 0) s_bad = p0 + j + 1;
      if (bad) break;  // the same in every thread
      if (mine && dk == j) {
        const double q = fast_rsqrt(d);
        if (di == j) {  // (the block keeps the pivot, which other threads may still read)
          c = mk<S>(sqrt_from(d, q), 0.0);
          rdb[j] = q;
        } else {
          Lb[j * LP + di] = c = cscale(c, q);
        }
      }
      __syncthreads();
      if ((tid >> 5) < nwt) {
        if (mine && dk > j) {
          c = cfms(Lb[j * LP + di], conjd(Lb[j * LP + dk]), c);
          if (di == dk) Lb[dk * LP + di] = c;  // the pivots to come
        }
      }
      __syncthreads();
    }
    __syncthreads();
    if (s_bad) {
      if (T.rank() == 0) *P.info = s_bad;
      return false;
    }
    // 2. the rows below: column by column, the rest of the row updated with each finished column
    for (int rb = p0 + w + 4 * T.swrank(); rb < n; rb += 4 * T.wsize()) {
      const int i = rb + (lane & 3), cg = lane >> 2;  // columns cg and cg + 8
      S r0 = mk<S>(0.0, 0.0), r1 = r0;
      if (i < n) {
        if (cg < w) r0 = B[i + (size_t)(p0 + cg) * ld];
        if (cg + 8 < w) r1 = B[i + (size_t)(p0 + cg + 8) * ld];
      }
#pragma unroll
      for (int j = 0; j < W; ++j) {
        const S f = cscale(shfl_c(j < 8 ? r0 : r1, (lane & 3) | (j & 7) << 2), rdb[j]);
        if (j < 8) {
          if (cg == j) r0 = f;
          else if (cg > j) r0 = cfms(f, conjd(Lb[j * LP + cg]), r0);
          r1 = cfms(f, conjd(Lb[j * LP + cg + 8]), r1);
        } else {
          if (cg == j - 8) r1 = f;
          else if (cg > j - 8) r1 = cfms(f, conjd(Lb[j * LP + cg + 8]), r1);
        }
      }
      if (i < n) {
        if (cg < w) B[i + (size_t)(p0 + cg) * ld] = r0;
        if (cg + 8 < w) B[i + (size_t)(p0 + cg + 8) * ld] = r1;
      }
    }
    if (!T.sync()) return false;
    // (behind the barrier: every CTA has read the block that this overwrites)
    if (first_cta) {
      if (mine && di < w) B[(p0 + di) + (size_t)(p0 + dk) * ld] = c;
      for (int j = tid; j < w; j += blockDim.x) rd[p0 + j] = rdb[j];
    }
    // 3. the trailing lower triangle, order m: columns a and m - 1 - a together have `len` or fewer
    // blocks of 32 rows
    const int k0 = p0 + w, m = n - k0;
    if (m > 0) {
      const int pairs = (m + 1) / 2, len = (m + 31) / 32 + 2;
      for (int t = T.swrank(); t < pairs * len; t += T.wsize()) {
        const int a = t / len;
        int q = t - a * len, k = k0 + a;
        const int na = (n - k + 31) / 32;
        if (q >= na) {
          q -= na;
          k = n - 1 - a;
          if (k == k0 + a) continue;  // the middle column of an odd order
        }
        const int i = k + 32 * q + lane;
        if (k + 32 * q >= n) continue;
        S f[W];
        const S mf = lane < W ? conjd(B[k + (size_t)(p0 + lane) * ld]) : mk<S>(0.0, 0.0);
        S v[W];
#pragma unroll
        for (int j = 0; j < W; ++j) v[j] = i < n ? B[i + (size_t)(p0 + j) * ld] : mk<S>(0.0, 0.0);
#pragma unroll
        for (int j = 0; j < W; ++j) f[j] = shfl_c(mf, j);
        S a0 = mk<S>(0.0, 0.0), a1 = a0;
#pragma unroll
        for (int j = 0; j < W; j += 2) {
          a0 = cfma(v[j], f[j], a0);
          a1 = cfma(v[j + 1], f[j + 1], a1);
        }
        if (i < n) B[i + (size_t)k * ld] = csub(B[i + (size_t)k * ld], cadd(a0, a1));
      }
      if (!T.sync()) return false;
    }
  }
  return T.sync();
}

// x <- L^{-1} x for one column x (stride 1) by the calling warp, in blocks of 32 rows: the
// diagonal block is solved in registers (lane l holds row b0 + l, values pass by shuffles), then the
// rows below are updated by a block product whose loads are all independent.  rd: 1 / L[i][i].
template <class S>
__device__ __forceinline__ void forward_subst(const S* __restrict__ L, const double* __restrict__ rd,
                                              int ld, int n, S* __restrict__ x) {
  const int lane = threadIdx.x & 31;
  for (int b0 = 0; b0 < n; b0 += 32) {
    const int bn = min(32, n - b0);
    S xl = lane < bn ? x[b0 + lane] : mk<S>(0.0, 0.0);
    const double rl = lane < bn ? rd[b0 + lane] : 0.0;
    for (int i = 0; i < bn; ++i) {
      if (lane == i) xl = cscale(xl, rl);
      const S xi = shfl_c(xl, i);
      if (lane > i && lane < bn) xl = cfms(L[(size_t)(b0 + i) * ld + b0 + lane], xi, xl);
    }
    if (lane < bn) x[b0 + lane] = xl;
    // rows below, two 32-row blocks per pass (every broadcast x_i serves both), eight columns of L
    // loaded ahead of their products: a warp has a quarter of the SM's FP64 pipe nearly to itself, and
    // what it waits for memory is lost
    for (int r0 = b0 + bn; r0 < n; r0 += 64) {
      const int r = r0 + lane, r2 = r + 32;
      const bool two = r0 + 32 < n;
      const S* lp = L + (size_t)b0 * ld + r;
      S a0 = mk<S>(0.0, 0.0), a1 = a0, c0 = a0, c1 = a0;
      int i = 0;
#pragma unroll 2
      for (; i + 8 <= bn; i += 8) {
        S l[8], m[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          l[u] = r < n ? lp[(size_t)(i + u) * ld] : mk<S>(0.0, 0.0);
          m[u] = r2 < n ? lp[(size_t)(i + u) * ld + 32] : mk<S>(0.0, 0.0);
        }
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
          const S xi = shfl_c(xl, i + u), xj = shfl_c(xl, i + u + 1);
          a0 = cfma(l[u], xi, a0);
          a1 = cfma(l[u + 1], xj, a1);
          if (two) {
            c0 = cfma(m[u], xi, c0);
            c1 = cfma(m[u + 1], xj, c1);
          }
        }
      }
      for (; i < bn; ++i) {
        const S xi = shfl_c(xl, i);
        if (r < n) a0 = cfma(lp[(size_t)i * ld], xi, a0);
        if (r2 < n) c0 = cfma(lp[(size_t)i * ld + 32], xi, c0);
      }
      if (r < n) x[r] = csub(x[r], cadd(a0, a1));
      if (r2 < n) x[r2] = csub(x[r2], cadd(c0, c1));
    }
  }
}

// x <- L^{-H} x for one column x by the calling warp, in blocks of 32 rows from the bottom: the
// diagonal block of L^H is solved in registers, then the rows above are updated (lane i reads the
// contiguous segment L[b0..b1), i] of column i).
template <class S>
__device__ __forceinline__ void backward_subst_h(const S* __restrict__ L, const double* __restrict__ rd,
                                                 int ld, int n, S* __restrict__ x) {
  const int lane = threadIdx.x & 31;
  for (int b1 = n; b1 > 0; b1 -= 32) {
    const int b0 = max(0, b1 - 32), bn = b1 - b0;
    S xl = lane < bn ? x[b0 + lane] : mk<S>(0.0, 0.0);
    const double rl = lane < bn ? rd[b0 + lane] : 0.0;
    for (int i = bn - 1; i >= 0; --i) {
      if (lane == i) xl = cscale(xl, rl);
      const S xi = shfl_c(xl, i);
      if (lane < i) xl = csub(xl, cmulc(L[(size_t)(b0 + lane) * ld + b0 + i], xi));
    }
    if (lane < bn) x[b0 + lane] = xl;
    // rows above, as below in the forward form (lane r reads the contiguous segment of column r)
    for (int r0 = 0; r0 < b0; r0 += 64) {
      const int r = r0 + lane, r2 = r + 32;
      const bool two = r0 + 32 < b0;
      S a0 = mk<S>(0.0, 0.0), a1 = a0, c0 = a0, c1 = a0;
      const S* lr = L + (size_t)r * ld + b0;
      const S* lr2 = lr + (size_t)32 * ld;
      int t = 0;
#pragma unroll 2
      for (; t + 8 <= bn; t += 8) {
        S l[8], m[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          l[u] = r < b0 ? lr[t + u] : mk<S>(0.0, 0.0);
          m[u] = r2 < b0 ? lr2[t + u] : mk<S>(0.0, 0.0);
        }
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
          const S xt = shfl_c(xl, t + u), xu = shfl_c(xl, t + u + 1);
          a0 = cfmac(l[u], xt, a0);
          a1 = cfmac(l[u + 1], xu, a1);
          if (two) {
            c0 = cfmac(m[u], xt, c0);
            c1 = cfmac(m[u + 1], xu, c1);
          }
        }
      }
      for (; t < bn; ++t) {
        const S xt = shfl_c(xl, t);
        if (r < b0) a0 = cfmac(lr[t], xt, a0);
        if (r2 < b0) c0 = cfmac(lr2[t], xt, c0);
      }
      if (r < b0) x[r] = csub(x[r], cadd(a0, a1));
      if (r2 < b0) x[r2] = csub(x[r2], cadd(c0, c1));
    }
  }
}

// ---- phase 2: C = L^{-1} A L^{-H} ---------------------------------------------------------------
template <class Team, class S>
__device__ bool reduce_standard(const Team& T, const Pencil<S>& P) {
  const int n = P.n, la = P.lda;
  S* A = P.A;
  S* R = P.R;
  const int lane = threadIdx.x & 31;
  // full Hermitian A from its lower triangle
  for (int i = T.swrank(); i < n; i += T.wsize()) {
    S* ci = A + (size_t)i * la;
    for (int j = lane; j < i; j += 32) ci[j] = conjd(A[i + (size_t)j * la]);
    if (lane == 0) ci[i] = mk<S>(re(ci[i]), 0.0);
  }
  if (!T.sync()) return false;
  // X = L^{-1} A, column by column, in place in A
  for (int c = T.swrank(); c < n; c += T.wsize()) forward_subst(P.B, vrdiag(P), P.ldb, n, A + (size_t)c * la);
  if (!T.sync()) return false;
  // R = X^H
  for (int r = T.swrank(); r < n; r += T.wsize()) {
    S* cr = R + (size_t)r * n;
    for (int c = lane; c < n; c += 32) cr[c] = conjd(A[r + (size_t)c * la]);
  }
  if (!T.sync()) return false;
  // C = L^{-1} X^H = L^{-1} A L^{-H}, in place in R
  for (int c = T.swrank(); c < n; c += T.wsize()) forward_subst(P.B, vrdiag(P), P.ldb, n, R + (size_t)c * n);
  if (!T.sync()) return false;
  // A = C, made exactly Hermitian (lower triangle kept, upper = its conjugate, real diagonal)
  for (int c = T.swrank(); c < n; c += T.wsize()) {
    S* ac = A + (size_t)c * la;
    for (int r = lane; r < n; r += 32) {
      S v;
      if (r > c) v = R[r + (size_t)c * n];
      else if (r < c) v = conjd(R[c + (size_t)r * n]);
      else v = mk<S>(re(R[c + (size_t)c * n]), 0.0);
      ac[r] = v;
    }
  }
  return T.sync();
}

// ---- phase 3: Householder tridiagonalisation ------------------------------------------------------
// vec layout: d[n], e[n], tau[2n] (n words of S), p[4n] (2 n words of S: p of two consecutive
// steps), 1/L_jj[n], q[2n] (Re conj(C v) v of two consecutive steps, complex pencils)
template <class S>
__device__ __forceinline__ double* vd(const Pencil<S>& P) { return P.vec; }
template <class S>
__device__ __forceinline__ double* ve(const Pencil<S>& P) { return P.vec + P.n; }
template <class S>
__device__ __forceinline__ S* vtau(const Pencil<S>& P) { return reinterpret_cast<S*>(P.vec + 2 * P.n); }
template <class S>
__device__ __forceinline__ S* vp(const Pencil<S>& P) { return reinterpret_cast<S*>(P.vec + 4 * P.n); }
template <class S>
__device__ __forceinline__ double* vq(const Pencil<S>& P) { return P.vec + 9 * P.n; }

// Sum over the CTA (every thread passes a value; every thread gets the same total, reduced in a
// fixed order so that all CTAs of a grid team obtain bit-identical results).
template <class S>
__device__ __forceinline__ S cta_sum_c(S v) {
  __shared__ S red[kWarps];
  v = warp_sum_c(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  // second level: the kWarps warp totals in every group of kWarps lanes, a butterfly within the
  // group (every lane ends with the same value: each level adds the same two operands, in either
  // order); the launch has kThreads threads
  S s = red[threadIdx.x & (kWarps - 1)];
#pragma unroll
  for (int o = kWarps / 2; o > 0; o >>= 1) s = cadd(s, shfl_xor_c(s, o));
  return s;
}

// Reflector j from x = column j of the updated matrix, rows j+1..n-1, staged in sx[j+1..n-1] by the
// whole CTA: beta = -sign(Re x_0) |x| (the real subdiagonal e_j), tau = (beta - x_0) / beta and
// v = x / (x_0 - beta) with v_{j+1} = 1, left in sx.  Every CTA of a grid team computes it the same
// way (fixed-order sums); the writer CTA also stores e_j, tau_j and v (column j of R).
template <class S>
__device__ S cta_reflector(const Pencil<S>& P, int j, S* sx, bool writer) {
  __shared__ S s_tau, s_vs;
  const int n = P.n, tid = threadIdx.x;
  __syncthreads();  // sx was staged by other threads
  double s = 0.0;
  for (int i = j + 2 + tid; i < n; i += blockDim.x) s = abs2_acc(sx[i], s);
  s = cta_sum_c(s);  // (its barriers also publish sx)
  if (tid == 0) {
    // one thread's chain: the signs and the zero test on the bits, not in FP64
    const S alpha = sx[j + 1];
    double beta;
    S tj = mk<S>(0.0, 0.0), vs = mk<S>(0.0, 0.0);
    if (((unsigned long long)dbits(s) << 1) == 0 && im(alpha) == 0.0) {
      beta = re(alpha);  // nothing to annihilate: H = I
    } else {
      const double a2 = abs2_acc(alpha, s);
      const double ra = fast_rsqrt(a2), an = sqrt_from(a2, ra);
      const bool pos = dbits(re(alpha)) >= 0;
      beta = pos ? -an : an;
      const S diff = mk<S>(re(alpha) - beta, im(alpha));  // v_i = x_i / (alpha - beta)
      vs = cinv(diff);
      tj = cscale(diff, pos ? ra : -ra);  // (beta - alpha) / beta
    }
    s_tau = tj;
    s_vs = vs;
    if (writer) {
      ve(P)[j] = beta;
      vtau(P)[j] = tj;
    }
  }
  __syncthreads();
  const S vs = s_vs, tj = s_tau;
  S* __restrict__ rj = P.R + (size_t)j * n;
  for (int i = j + 1 + tid; i < n; i += blockDim.x) {
    const S v = i == j + 1 ? mk<S>(1.0, 0.0) : cmul(sx[i], vs);
    sx[i] = v;
    if (writer) rj[i] = v;
  }
  __syncthreads();
  return tj;
}

// One pass over this CTA's columns k >= kmin, rows >= r0, by all its warps: with UPDATE the rank-2 update
// C <- C - v w^H - w v^H; then u_k = (column k)^H vn (C is Hermitian: row k of C vn), from which
// pn[k] = tn u_k and, for complex pencils, qn[k] = Re conj(u_k) vn_k are stored.  Column k belongs to CTA
// k mod G.  The columns' blocks of 32 rows, one column after another, are cut into equal shares for
// the warps, so that none of the SM's FP64 quarters idles when few columns are left; the sums of a
// column that is cut go through shared memory.  kout: the column whose update goes to global memory
// (the next one to be eliminated, which every CTA reads); the others stay where they are.
template <bool UPDATE, class Team, class S>
__device__ void column_pass(const Team& T, const Pencil<S>& P, S* cols, bool resident, int kmin, int r0, int kout,
                            const S* sv, const S* sw, const S* sn, S tn, S* __restrict__ pn, double* __restrict__ qn) {
  __shared__ S s_start[kWarps], s_head[kWarps];
  __shared__ int s_k[kWarps], s_last[kWarps];
  const int n = P.n, G = T.ctas(), cta = T.cta();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int slots = cta < n ? (n - cta + G - 1) / G : 0;
  const int s0 = kmin > cta ? (kmin - cta + G - 1) / G : 0;
  const int cnt = max(slots - s0, 0), nch = (n - r0 + 31) / 32, tot = cnt * nch;
  auto put = [&](int k, S u) {
    pn[k] = cmul(tn, u);
    if constexpr (sizeof(S) == sizeof(double2)) qn[k] = re(cmulc(u, sn[k]));
  };
  int lo = warp * tot / kWarps;
  const int hi = (warp + 1) * tot / kWarps;
  if (lane == 0) {
    s_k[warp] = -1;
    s_head[warp] = mk<S>(0.0, 0.0);  // (a share may be empty)
  }
  while (lo < hi) {
    const int c = lo / nch, ch = lo - c * nch, end = min(nch, ch + hi - lo);
    const int k = (s0 + c) * G + cta;
    S cvk = mk<S>(0.0, 0.0), cwk = cvk;
    if (UPDATE) {
      cvk = conjd(sv[k]);
      cwk = conjd(sw[k]);
    }
    S* gk = P.A + (size_t)k * P.lda;
    S* ck = resident ? cols + (size_t)(s0 + c) * n : gk;
    S* dst = k == kout ? gk : ck;
    S acc = mk<S>(0.0, 0.0);
    const int iend = min(n, r0 + 32 * end);
    int i = r0 + 32 * ch + lane;
    for (; i + 96 < iend; i += 128) {
      S a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = ck[i + 32 * u];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = i + 32 * u;
        if (UPDATE) {
          a[u] = cfms(sw[r], cvk, cfms(sv[r], cwk, a[u]));
          dst[r] = a[u];
        }
        acc = cfmac(a[u], sn[r], acc);
      }
    }
    for (; i < iend; i += 32) {
      S a = ck[i];
      if (UPDATE) {
        a = cfms(sw[i], cvk, cfms(sv[i], cwk, a));
        dst[i] = a;
      }
      acc = cfmac(a, sn[i], acc);
    }
    acc = warp_sum_c(acc);
    if (lane == 0) {
      if (ch == 0 && end == nch) {
        put(k, acc);
      } else if (ch == 0) {  // to be continued by the next warps
        s_start[warp] = acc;
        s_k[warp] = k;
        s_last[warp] = ((c + 1) * nch * kWarps - 1) / tot;  // the warp with the column's last block
      } else {
        s_head[warp] = acc;
      }
    }
    lo += end - ch;
  }
  __syncthreads();
  if (tid < kWarps && s_k[tid] >= 0) {
    S u = s_start[tid];
    for (int q = tid + 1; q <= s_last[tid]; ++q) u = cadd(u, s_head[q]);
    put(s_k[tid], u);
  }
}

// One team barrier per column.  Step j applies reflector j (v_j, tau_j, and p_j = tau_j C v_j from
// the previous step) to the trailing matrix: gamma = -(tau_j / 2) p_j^H v_j (real: v_j^H C v_j is, so a
// complex pencil adds up the real parts q_j that come with p_j), w = p_j + gamma v_j,
// C <- C - v w^H - w v^H.  Every CTA forms column j+1 of the updated matrix and reflector j+1 from
// it in shared memory (the same values in every CTA), then updates its columns k >= j+2
// and, in the same pass over the column, accumulates p_{j+1}[k] (column_pass).  Rows < j+2 of those
// columns are never read again and are not updated.  p of consecutive steps alternate between two
// buffers, so that a CTA still reading p_j never meets the p_{j+1} that faster CTAs write.
// What bounds it: per step two barrier and L2 round trips, about 30 dependent FP64 operations of 64 to
// 100 cycles each, and the update's FP64 instructions.  The CTA's columns therefore stay in shared
// memory when they fit, and the update is spread evenly over the SM (column_pass).  Cycles per step
// (load, reflector and barrier / update), order 564 complex: 14.6k / 7.7k (columns in L2, a warp a column: 15.9k
// / 12.1k); 1127 real: 11.9k / 7.5k (13.9k / 8.8k).
// sbuf: 3 n words of S of shared memory per CTA (v_j, w and v_{j+1}, indexed by row), then, when
// P.resident, the CTA's columns.
template <class Team, class S>
__device__ bool tridiagonalise(const Team& T, const Pencil<S>& P, S* sbuf) {
  constexpr bool kComplex = sizeof(S) == sizeof(double2);
  const int n = P.n, la = P.lda;
  S* A = P.A;
  const int tid = threadIdx.x;
  const bool writer = T.rank() < (int)blockDim.x;  // the first CTA writes d, e, tau and R
  if (n == 1) {
    if (T.rank() == 0) vd(P)[0] = re(A[0]);
    return T.sync();
  }
  S* sv = sbuf;
  S* sw = sbuf + n;
  S* sn = sbuf + 2 * n;
  S* cols = sbuf + 3 * n;
  const bool resident = P.resident != 0;
  if (resident) {
    for (int s = 0, k = T.cta(); k < n; ++s, k += T.ctas())
      for (int i = tid; i < n; i += blockDim.x) cols[(size_t)s * n + i] = A[i + (size_t)k * la];
  }
  // reflector 0 from column 0, and p_0 = tau_0 C v_0 (rows 1..n-1)
  for (int i = 1 + tid; i < n; i += blockDim.x) sv[i] = A[i];
  if (writer && tid == 0) vd(P)[0] = re(A[0]);
  S tau = cta_reflector(P, 0, sv, writer);
  column_pass<false>(T, P, cols, resident, 1, 1, -1, sv, sv, sv, tau, vp(P), vq(P));
  if (!T.sync()) return false;
  for (int j = 0; j <= n - 2; ++j) {
    const S* pj = vp(P) + (size_t)(j & 1) * n;
    const double* qj = vq(P) + (size_t)(j & 1) * n;
    // p_j and column j+1 of C are read together (one round trip to L2), staged raw in sw and sn;
    // then w = p_j + gamma v_j and column j+1 of the updated matrix, x - v conj(w_{j+1}) - w (the
    // entry of v_j in row j+1 is 1), each thread on its own rows
    const S* c1 = A + (size_t)(j + 1) * la;
    double g = 0.0;
    for (int i = j + 1 + tid; i < n; i += blockDim.x) {
      const S pi = pj[i];
      if constexpr (kComplex) g += qj[i];
      else g = fma(pi, sv[i], g);
      sn[i] = c1[i];
      sw[i] = pi;
    }
    g = cta_sum_c(g);
    double gamma;  // -|tau|^2 v^H C v / 2
    if constexpr (kComplex) gamma = -0.5 * g * abs2_acc(tau, 0.0);
    else gamma = -0.5 * g * tau;
    auto wof = [&](S p, S v) {
      if constexpr (kComplex) return make_double2(fma(gamma, v.x, p.x), fma(gamma, v.y, p.y));
      else return fma(gamma, v, p);
    };
    const S cw1 = conjd(wof(pj[j + 1], mk<S>(1.0, 0.0)));
    for (int i = j + 1 + tid; i < n; i += blockDim.x) {
      const S wi = wof(sw[i], sv[i]);
      const S x = csub(cfms(sv[i], cw1, sn[i]), wi);
      sw[i] = wi;
      sn[i] = x;
      if (i == j + 1 && writer) vd(P)[j + 1] = re(x);
    }
    if (j + 1 <= n - 2) {
      const S tn = cta_reflector(P, j + 1, sn, writer);
      column_pass<true>(T, P, cols, resident, j + 2, j + 2, j + 2, sv, sw, sn, tn, vp(P) + (size_t)((j + 1) & 1) * n,
                        vq(P) + (size_t)((j + 1) & 1) * n);
      tau = tn;
    }
    if (!T.sync()) return false;
    S* t = sv;  // v_{j+1} becomes the current reflector
    sv = sn;
    sn = t;
  }
  return true;
}

// ---- phase 4: eigenpairs of the symmetric tridiagonal T (d, e) -----------------------------------
// The phase works on T scaled by a power of two to norm [1, 2), staged in shared memory as (d_i,
// e_{i-1}^2) pairs (and the same in FP32), later as (d_i, e_i).
//
// Number of eigenvalues of T below s, from the signs of the leading principal minors p_i of
// T - s I (a Sturm sequence): p_0 = 1, p_{i+1} = (d_i - s) p_i - e_{i-1}^2 p_{i-1} with e_{-1} = 0;
// the count is the number of sign changes between consecutive minors, i.e. of negative pivots
// p_{i+1} / p_i of the LDL^T factorisation (Sylvester's law of inertia).  Division-free: one fused
// multiply-add per row on the dependent chain (an FP64 division has about seven times the latency
// of a fused multiply-add on GB300, where that latency is already 64 cycles), and everything else
// beside it: rows go four at a time, whose minors are only checked to be of size 2^-400 to 2^400;
// the four rows are repeated one by one when they are not.  There the pair (p_i, p_{i+1}) is rescaled
// by an exact power of two when p_{i+1} leaves [2^-600, 2^600], and an exactly zero minor is
// replaced by -2^-600 times the previous one (a tiny negative pivot), which also carries the
// sequence across a split (e_i = 0).  The last minor is v 2^ve.
struct Sturm {
  int count, ve;
  double v;
};
// |x| as an integer: ordered like |x| for all non-NaN doubles
__device__ __forceinline__ unsigned long long dmag(double x) {
  return (unsigned long long)dbits(x) & 0x7FFFFFFFFFFFFFFFull;
}
// 2^e, the exponent taken into the normal range
__device__ __forceinline__ double exp2_of(int e) { return __hiloint2double((1023 + max(-1022, min(1023, e))) << 20, 0); }

__device__ __forceinline__ Sturm sturm_count(const double2* __restrict__ t, int n, double s) {
  double pm = 0.0, p = 1.0;
  int c = 0, es = 0;
  auto row = [&](double2 a) {  // one row with all the checks
    double pn = fma(a.x - s, p, -a.y * pm);
    if (((unsigned long long)dbits(pn) << 1) == 0) pn = -0x1p-600 * p;
    c += (int)((unsigned long long)(dbits(pn) ^ dbits(p)) >> 63);
    pm = p;
    p = pn;
    const int ex = (int)((dbits(p) >> 52) & 0x7FF);  // biased exponent of |p|
    if (ex > 1023 + 600) {
      p *= 0x1p-600;
      pm *= 0x1p-600;
      es += 600;
    } else if (ex < 1023 - 600 && (int)((dbits(pm) >> 52) & 0x7FF) < 1023 + 400) {
      p *= 0x1p+600;
      pm *= 0x1p+600;
      es -= 600;
    }
  };
  int i = 0;
  for (; i + 4 <= n; i += 4) {
    const double2 a0 = t[i], a1 = t[i + 1], a2 = t[i + 2], a3 = t[i + 3];
    const double q0 = fma(a0.x - s, p, -a0.y * pm);
    const double q1 = fma(a1.x - s, q0, -a1.y * p);
    const double q2 = fma(a2.x - s, q1, -a2.y * q0);
    const double q3 = fma(a3.x - s, q2, -a3.y * q1);
    const int h = __double2hiint(p), h0 = __double2hiint(q0), h1 = __double2hiint(q1), h2 = __double2hiint(q2),
              h3 = __double2hiint(q3);
    auto out = [](int x) { return (unsigned)((x & 0x7ff00000) - ((1023 - 400) << 20)) > (unsigned)(800 << 20); };
    if (out(h0) | out(h1) | out(h2) | out(h3)) {
#pragma unroll 1
      for (int u = 0; u < 4; ++u) row(t[i + u]);
      continue;
    }
    c += ((unsigned)(h ^ h0) >> 31) + ((unsigned)(h0 ^ h1) >> 31) + ((unsigned)(h1 ^ h2) >> 31) +
         ((unsigned)(h2 ^ h3) >> 31);
    pm = q2;
    p = q3;
    const int ex = ((h3 >> 20) & 0x7FF) - 1023;
    if (ex > 200 || ex < -200) {
      const double f = exp2_of(-ex);
      p *= f;
      pm *= f;
      es += ex;
    }
  }
  for (; i < n; ++i) row(t[i]);
  return Sturm{c, es, p};
}
// The same count in FP32 (about 64 times cheaper on GB300), used only to narrow the bracket.
__device__ __forceinline__ int sturm_count32(const float2* __restrict__ t, int n, float s, float pivmin) {
  int c = 0;
  float q = 1.f;
#pragma unroll 4
  for (int i = 0; i < n; ++i) {
    const float2 a = t[i];
    q = (a.x - s) - __fdividef(a.y, q);
    if (fabsf(q) < pivmin) q = -pivmin;
    c += q < 0.f;
  }
  return c;
}

// Deterministic start vector entry in (-1, 1) for eigenvector k, row i.
__device__ __forceinline__ double start_entry(int k, int i) {
  unsigned h = (unsigned)k * 0x9E3779B1u ^ ((unsigned)i + 0x7F4A7C15u) * 0x85EBCA77u;
  h ^= h >> 16;
  h *= 0x7FEB352Du;
  h ^= h >> 15;
  h *= 0x846CA68Bu;
  h ^= h >> 16;
  return ((double)(h >> 8) + 0.5) * (2.0 / 16777216.0) - 1.0;
}

// smem: 3 n words of S
template <class Team, class S>
__device__ bool tridiagonal_eig(const Team& T, const Pencil<S>& P, S* smem) {
  const int n = P.n;
  const double* d = vd(P);
  const double* e = ve(P);
  double* w = P.w;
  const int tid = threadIdx.x, lane = tid & 31;
  double2* t64 = reinterpret_cast<double2*>(smem);
  float2* t32 = reinterpret_cast<float2*>(t64 + n);
  // norm and Gershgorin interval (every warp computes them the same way, in the scaled units below)
  double tn = 0.0, glo = 1e308, gu = -1e308;
  for (int i = lane; i < n; i += 32) {
    const double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + (i < n - 1 ? fabs(e[i]) : 0.0);
    tn = fmax(tn, fabs(d[i]) + r);
    glo = fmin(glo, d[i] - r);
    gu = fmax(gu, d[i] + r);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
    glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
    gu = fmax(gu, __shfl_xor_sync(0xffffffffu, gu, o));
  }
  tn = fmax(tn, 1e-300);
  const int tex = max(-1000, min(1000, (int)(dbits(tn) >> 52 & 0x7FF) - 1023));
  const double sc = exp2_of(-tex), usc = exp2_of(tex);
  const double eps = 2.220446049250313e-16;
  tn *= sc;
  glo = glo * sc - 2.0 * eps * tn;
  gu = gu * sc + 2.0 * eps * tn;
  for (int i = tid; i < n; i += blockDim.x) {
    const double di = d[i] * sc, ei = i > 0 ? e[i - 1] * sc : 0.0;
    t64[i] = make_double2(di, ei * ei);
    t32[i] = make_float2((float)di, (float)(ei * ei));
  }
  __syncthreads();
  // Eigenvalue k by a group of kSect lanes.  A bracket [lo, hi] (count(lo) <= k < count(hi)) is first
  // narrowed with FP32 counts to 1e-6 |T|, widened by 2e-6 |T| and accepted only if the FP64
  // counts at both ends confirm it (else the Gershgorin interval is used); FP64 rounds take it to
  // 2 eps |lambda|.  In every round each lane of the group counts at one point of the bracket and
  // the bracket becomes the interval between the last point below the eigenvalue and the first
  // above it.  While the bracket holds a single eigenvalue the points stand at geometric distances
  // on both sides of the root that the last minors at its ends interpolate (regula falsi): at each
  // round the bracket shrinks to about its square over the distance to the next eigenvalue, three
  // or four rounds from 4e-6 |T| where even sections take about ten.  A round that gains less than a
  // factor 8, or a bracket with several eigenvalues, is followed by one with evenly spaced points.
  // Orders 564 and 1127: 0.75 and 1.49 ms (even sections, unblocked counts: 2.08 and 4.66).
  const float pivmin32 = 1e-30f;
  // 8 lanes an eigenvalue, 4 where that would keep the team's FP64 units busy for several passes
  const int kSect = T.size() >= 8 * n ? 8 : 4;
  const int kGroups = 32 / kSect;
  {
    const int grp = lane / kSect, gi = lane % kSect, g0 = grp * kSect;
    const unsigned gmask = ((1u << kSect) - 1u) << g0;
    auto first_above = [&](bool above) {
      const unsigned bits = (__ballot_sync(0xffffffffu, above) & gmask) >> g0;
      return bits ? __ffs(bits) - 1 : kSect;
    };
    for (int k0 = T.swrank() * kGroups; k0 < n; k0 += T.wsize() * kGroups) {
      const int k = k0 + grp;
      const bool act = k < n;
      float l32 = (float)glo, h32 = (float)gu;
      const float wid = (float)(1e-6 * tn);
      bool open = act;
      for (int it = 0; it < 24; ++it) {
        open = open && h32 - l32 > wid;
        if (!__any_sync(0xffffffffu, open)) break;
        const float step = (h32 - l32) * (1.0f / (float)(kSect + 1));
        const float pt = l32 + (float)(gi + 1) * step;
        const int f = first_above(open && pt < h32 && sturm_count32(t32, n, pt, pivmin32) > k);
        if (open) {
          const float nl = f == 0 ? l32 : l32 + (float)f * step;
          const float nh = f == kSect ? h32 : l32 + (float)(f + 1) * step;
          if (nh > nl) {
            l32 = nl;
            h32 = fminf(nh, h32);
          } else {
            open = false;
          }
        }
      }
      double lo = fmax(glo, (double)l32 - 2e-6 * tn), hi = fmin(gu, (double)h32 + 2e-6 * tn);
      Sturm flo{0, 0, 0.0}, fhi{0, 0, 0.0};
      {
        Sturm c{0, 0, 0.0};
        if (act && gi < 2) c = sturm_count(t64, n, gi ? hi : lo);
        flo.count = __shfl_sync(0xffffffffu, c.count, g0);
        flo.ve = __shfl_sync(0xffffffffu, c.ve, g0);
        flo.v = __shfl_sync(0xffffffffu, c.v, g0);
        fhi.count = __shfl_sync(0xffffffffu, c.count, g0 + 1);
        fhi.ve = __shfl_sync(0xffffffffu, c.ve, g0 + 1);
        fhi.v = __shfl_sync(0xffffffffu, c.v, g0 + 1);
        if (!(flo.count <= k && fhi.count > k)) {
          lo = glo;
          hi = gu;
          flo = Sturm{0, 0, 0.0};
          fhi = Sturm{n, 0, 0.0};
        }
      }
      open = act;
      bool even = false;  // this round takes evenly spaced points
      for (int it = 0; it < 80; ++it) {
        open = open && !(hi - lo <= 2.0 * eps * fmax(fabs(lo), fabs(hi)) + 1e-300);
        if (!__any_sync(0xffffffffu, open)) break;
        const double width = hi - lo;
        // (a count of 0 or n at the ends of the Gershgorin interval comes without its minor)
        const bool ladder = !even && fhi.count - flo.count == 1 && flo.v != 0.0 && fhi.v != 0.0;
        double pt;
        if (ladder) {
          const double r = fabs(fhi.v) * exp2_of(fhi.ve - flo.ve) * fast_rcp(fabs(flo.v));
          const double est = lo + width * fast_rcp(1.0 + r);
          const int half = kSect >> 1, j = gi < half ? gi : kSect - 1 - gi;  // 0: outermost
          // exponents of the distances: 3, 8, 14, 22 below the bracket's width (two lanes a side: 6, 16)
          const int down = kSect == 8 ? (j == 0 ? 3 : j == 1 ? 8 : j == 2 ? 14 : 22) : (j == 0 ? 6 : 16);
          const double del = fmax(width * exp2_of(-down), 0.95 * eps * fabs(est));
          pt = gi < half ? est - del : est + del;
        } else {
          pt = lo + (double)(gi + 1) * (width * (1.0 / (double)(kSect + 1)));
        }
        Sturm c{0, 0, 0.0};
        const bool in = open && pt > lo && pt < hi;
        if (in) c = sturm_count(t64, n, pt);
        const int f = first_above(in ? c.count > k : !(pt <= lo));
        const int sl = g0 + max(f - 1, 0), sh = g0 + min(f, kSect - 1);
        const double pl = __shfl_sync(0xffffffffu, pt, sl), ph = __shfl_sync(0xffffffffu, pt, sh);
        const Sturm cl{__shfl_sync(0xffffffffu, c.count, sl), __shfl_sync(0xffffffffu, c.ve, sl),
                       __shfl_sync(0xffffffffu, c.v, sl)};
        const Sturm ch{__shfl_sync(0xffffffffu, c.count, sh), __shfl_sync(0xffffffffu, c.ve, sh),
                       __shfl_sync(0xffffffffu, c.v, sh)};
        if (open) {
          if (f > 0 && pl > lo) {
            lo = pl;
            flo = cl;
          }
          if (f < kSect && ph < hi) {
            hi = ph;
            fhi = ch;
          }
          const double nw = hi - lo;
          if (!(nw < width)) {
            if (!ladder) open = false;  // the points have become neighbours
            even = true;
          } else {
            even = ladder && nw > 0.125 * width;
          }
        }
      }
      if (act && gi == 0) w[k] = 0.5 * (lo + hi) * usc;
    }
  }
  if (!T.sync()) return false;
  T.stamp(4);
  // Eigenvectors by inverse iteration, one cluster per thread, in the scaled units.  T - s I = P L U
  // (partial pivoting) once, then two solves for a single eigenvalue, four for each of a cluster; the
  // first solve starts behind L (a random vector stays random).  With the eigenvalue good to
  // 2 eps |T| and the next one 1e-5 |T| away, one solve leaves about 1e-10 of the other vectors and
  // the second nothing.  Orders 564 and 1127: 0.81 and 1.60 ms (three full solves, row by row: 2.07 and
  // 4.85).  A chain of n dependent rows per pass, so every pass reads its arrays
  // eight rows ahead and keeps all but one multiply-add a row off the chain: the diagonal of U is
  // stored as reciprocals, already multiplied into its first superdiagonal.
  for (int i = tid; i < n; i += blockDim.x) t64[i] = make_double2(d[i] * sc, i < n - 1 ? e[i] * sc : 0.0);
  __syncthreads();
  const double ortol = 1e-5 * tn * usc;
  const double tiny = eps * tn;
  const size_t nn = (size_t)n * n;
  double* __restrict__ ua = P.wk;           // reciprocals of U's diagonal
  double* __restrict__ ub = P.wk + nn;      // U first superdiagonal over its diagonal
  double* __restrict__ ml = P.wk + 2 * nn;  // multipliers
  double* __restrict__ x = P.wk + 3 * nn;   // iterate
  double* __restrict__ y = P.wk + 4 * nn;   // L^{-1} P x
  unsigned* __restrict__ sw = reinterpret_cast<unsigned*>(P.wk + 5 * nn);  // bit i: rows i, i+1 swapped
  constexpr int U = 8;  // rows a block
  // 32 consecutive eigenvalues per warp (the interleaved arrays are then read in full 256-byte
  // rows), the warps spread over the CTAs
  for (int k0 = T.swrank() * 32 + lane; k0 < n; k0 += T.size()) {
    if (k0 > 0 && w[k0] - w[k0 - 1] <= ortol) continue;  // not the first of its cluster
    int k1 = k0 + 1;
    while (k1 < n && w[k1] - w[k1 - 1] <= ortol) ++k1;
    double sprev = 0.0;
    for (int m = k0; m < k1; ++m) {
      // slot m of the interleaved arrays: element i at [i * n + m]
      double s = w[m] * sc;
      const double pert = 10.0 * eps * fmax(fabs(s), tn);
      if (m > k0 && s - sprev < pert) s = sprev + pert;
      sprev = s;
      {
        double2 ti = t64[0];
        double a = ti.x - s, b = ti.y;
        unsigned bits = 0;
        for (int i = 0; i < n - 1; ++i) {
          const double2 tj = t64[i + 1];
          const double sub = ti.y, nd = tj.x - s, ns = tj.y;
          const size_t o = (size_t)i * n + m;
          // the pivot choice compares magnitudes as integers (the FP64 compare would add 64 cycles a
          // row); a pivot below eps |T| is taken as that
          const bool swp = dmag(a) < dmag(sub);
          double piv = swp ? sub : a;
          if (dmag(piv) < dmag(tiny)) piv = tiny;
          const double r = fast_rcp(piv), l = (swp ? a : sub) * r;
          ua[o] = r;
          ub[o] = (swp ? nd : b) * r;
          ml[o] = l;
          bits |= (unsigned)swp << (i & 31);
          if ((i & 31) == 31 || i == n - 2) {
            sw[(size_t)(i >> 5) * n + m] = bits;
            bits = 0;
          }
          a = swp ? fma(-l, nd, b) : fma(-l, b, nd);
          b = swp ? -l * ns : ns;
          ti = tj;
        }
        if (dmag(a) < dmag(tiny)) a = tiny;
        ua[(size_t)(n - 1) * n + m] = fast_rcp(a);
      }
      const bool cluster = k1 - k0 > 1;
      const int iters = cluster ? 4 : 2;
      for (int it = 0; it < iters; ++it) {
        // forward: y = L^{-1} P x, the row operations of the factorisation (running row in a register)
        if (it == 0) {
          for (int i = 0; i < n; ++i) y[(size_t)i * n + m] = start_entry(m, i);
        } else {
          double cur = x[m];
          unsigned bits = 0;
          int i = 0;
          for (; i + U <= n - 1; i += U) {
            double nx[U], l[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              nx[u] = x[(size_t)(i + u + 1) * n + m];
              l[u] = ml[(size_t)(i + u) * n + m];
            }
            if ((i & 31) == 0) bits = sw[(size_t)(i >> 5) * n + m];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const bool swp = bits >> ((i + u) & 31) & 1u;
              const double yv = swp ? nx[u] : cur, nv = swp ? cur : nx[u];
              y[(size_t)(i + u) * n + m] = yv;
              cur = fma(-l[u], yv, nv);
            }
          }
          for (; i < n - 1; ++i) {
            const size_t o = (size_t)i * n + m;
            const bool swp = sw[(size_t)(i >> 5) * n + m] >> (i & 31) & 1u;
            const double nx = x[o + n];
            const double yv = swp ? nx : cur, nv = swp ? cur : nx;
            y[o] = yv;
            cur = fma(-ml[o], yv, nv);
          }
          y[(size_t)(n - 1) * n + m] = cur;
        }
        // backward: x = U^{-1} y (the two solved rows below in registers; the iterate and the rows
        // still to solve are scaled down together when a block of rows has grown beyond 1e100)
        {
          double x1 = 0.0, x2 = 0.0;
          for (int i0 = n; i0 > 0; i0 -= U) {
            const int cnt = min(U, i0);
            double yv[U], uv[U], bv[U], cv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const int i = i0 - 1 - u;
              yv[u] = uv[u] = bv[u] = cv[u] = 0.0;
              if (u < cnt) {
                const size_t o = (size_t)i * n + m;
                yv[u] = y[o];
                uv[u] = ua[o];
                if (i < n - 1) {
                  bv[u] = ub[o];
                  // second superdiagonal (fill-in of a swap): e_{i+1}
                  if (sw[(size_t)(i >> 5) * n + m] >> (i & 31) & 1u) cv[u] = t64[i + 1].y;
                }
              }
            }
            unsigned long long big = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const double v = fma(-bv[u], x1, fma(-(cv[u] * uv[u]), x2, yv[u] * uv[u]));
              if (u < cnt) {
                x[(size_t)(i0 - 1 - u) * n + m] = v;
                x2 = x1;
                x1 = v;
                big = max(big, dmag(v));
              }
            }
            if (big > dmag(1e100)) {
              for (int r = 0; r < n; ++r) {
                if (r >= i0 - cnt) x[(size_t)r * n + m] *= 1e-100;
                else y[(size_t)r * n + m] *= 1e-100;
              }
              x1 *= 1e-100;
              x2 *= 1e-100;
            }
          }
        }
        if (!cluster && it + 1 < iters) continue;
        // orthogonalise against the cluster's earlier vectors, then normalise
        for (int q = k0; q < m; ++q) {
          const double* zq = P.Z + (size_t)q * n;
          double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
          int i = 0;
          for (; i + U <= n; i += U) {
            double z[U], v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              z[u] = zq[i + u];
              v[u] = x[(size_t)(i + u) * n + m];
            }
#pragma unroll
            for (int u = 0; u < U; u += 4) {
              s0 = fma(z[u], v[u], s0);
              s1 = fma(z[u + 1], v[u + 1], s1);
              s2 = fma(z[u + 2], v[u + 2], s2);
              s3 = fma(z[u + 3], v[u + 3], s3);
            }
          }
          for (; i < n; ++i) s0 = fma(zq[i], x[(size_t)i * n + m], s0);
          const double dot = (s0 + s1) + (s2 + s3);
          for (i = 0; i + U <= n; i += U) {
            double z[U], v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              z[u] = zq[i + u];
              v[u] = x[(size_t)(i + u) * n + m];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) x[(size_t)(i + u) * n + m] = fma(-dot, z[u], v[u]);
          }
          for (; i < n; ++i) x[(size_t)i * n + m] = fma(-dot, zq[i], x[(size_t)i * n + m]);
        }
        double n0 = 0.0, n1 = 0.0, n2 = 0.0, n3 = 0.0;  // four independent chains
        int i = 0;
        for (; i + U <= n; i += U) {
          double v[U];
#pragma unroll
          for (int u = 0; u < U; ++u) v[u] = x[(size_t)(i + u) * n + m];
#pragma unroll
          for (int u = 0; u < U; u += 4) {
            n0 = fma(v[u], v[u], n0);
            n1 = fma(v[u + 1], v[u + 1], n1);
            n2 = fma(v[u + 2], v[u + 2], n2);
            n3 = fma(v[u + 3], v[u + 3], n3);
          }
        }
        for (; i < n; ++i) {
          const double v = x[(size_t)i * n + m];
          n0 = fma(v, v, n0);
        }
        const double nrm = sqrt((n0 + n1) + (n2 + n3));
        const double r = nrm > 0.0 ? 1.0 / nrm : 0.0;
        double* __restrict__ zm = P.Z + (size_t)m * n;
        const bool last = it + 1 == iters;
        for (i = 0; i < n; i += U) {
          double v[U];
#pragma unroll
          for (int u = 0; u < U; ++u) v[u] = i + u < n ? x[(size_t)(i + u) * n + m] * r : 0.0;
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (i + u < n) {
              if (last) zm[i + u] = v[u];
              else x[(size_t)(i + u) * n + m] = v[u];
            }
        }
      }
    }
  }
  return T.sync();
}

// ---- phase 5: x = L^{-H} Q z ------------------------------------------------------------------
template <class Team, class S>
__device__ bool back_transform(const Team& T, const Pencil<S>& P, S* smem) {
  const int n = P.n;
  const int lane = threadIdx.x & 31;
  const S* tau = vtau(P);
  for (int c = T.swrank(); c < n; c += T.wsize()) {
    // The column is built in this warp's shared-memory slot when the launch provided one, else in
    // place in A's column c (A is free: the reflectors live in R, L in B).
    S* ac = P.A + (size_t)c * P.lda;
    S* vc = smem ? smem + (size_t)(threadIdx.x >> 5) * n : ac;
    const double* zc = P.Z + (size_t)c * n;
    for (int i = lane; i < n; i += 32) vc[i] = mk<S>(zc[i], 0.0);
    __syncwarp();
    // V = H_0 H_1 ... H_{n-2} Z: reflector j (rows j+1..n-1, stored in column j of R) applied last-first,
    // U 32-row blocks loaded ahead of their products; the first U of the next reflector while this one's
    // sum goes around the warp
    constexpr int U = sizeof(S) == sizeof(double) ? 8 : 4;
    S nx[U];
    auto first = [&](int j) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = j + 1 + lane + 32 * u;
        nx[u] = j >= 0 && i < n ? P.R[(size_t)j * n + i] : mk<S>(0.0, 0.0);
      }
    };
    first(n - 2);
    for (int j = n - 2; j >= 0; --j) {
      const S tj = tau[j];
      const S* rj = P.R + (size_t)j * n;
      S h[U];
#pragma unroll
      for (int u = 0; u < U; ++u) h[u] = nx[u];
      S s = mk<S>(0.0, 0.0), s2 = s;
      const int i0 = j + 1 + lane, m = n - 1 - j;  // rows of the reflector
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (32 * u < m) {
          if (u & 1) s2 = cfmac(h[u], i0 + 32 * u < n ? vc[i0 + 32 * u] : mk<S>(0.0, 0.0), s2);
          else s = cfmac(h[u], i0 + 32 * u < n ? vc[i0 + 32 * u] : mk<S>(0.0, 0.0), s);
        }
      for (int b = 32 * U; b < m; b += 32 * U) {
        S l[U];
#pragma unroll
        for (int u = 0; u < U; ++u) l[u] = i0 + b + 32 * u < n ? rj[i0 + b + 32 * u] : mk<S>(0.0, 0.0);
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (b + 32 * u < m) {
            const S v = i0 + b + 32 * u < n ? vc[i0 + b + 32 * u] : mk<S>(0.0, 0.0);
            if (u & 1) s2 = cfmac(l[u], v, s2);
            else s = cfmac(l[u], v, s);
          }
      }
      first(j - 1);
      s = cmul(tj, warp_sum_c(cadd(s, s2)));
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (32 * u < m && i0 + 32 * u < n) vc[i0 + 32 * u] = cfms(h[u], s, vc[i0 + 32 * u]);
      for (int b = 32 * U; b < m; b += 32 * U) {
        S l[U];
#pragma unroll
        for (int u = 0; u < U; ++u) l[u] = i0 + b + 32 * u < n ? rj[i0 + b + 32 * u] : mk<S>(0.0, 0.0);
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (b + 32 * u < m && i0 + b + 32 * u < n) vc[i0 + b + 32 * u] = cfms(l[u], s, vc[i0 + b + 32 * u]);
      }
      __syncwarp();  // (the next reflector's rows lie one lane further)
    }
    __syncwarp();
    backward_subst_h(P.B, vrdiag(P), P.ldb, n, vc);
    __syncwarp();
    // into the caller's complex A (in place for a complex pencil: the same lane, the same element)
    double2* oc = P.outA + (size_t)c * P.ldoa;
    for (int i = lane; i < n; i += 32) oc[i] = widen(vc[i]);
    __syncwarp();
  }
  return T.sync();
}

template <class Team, class S>
__device__ void solve_pencil(const Team& T, const Pencil<S>& P) {
  extern __shared__ double2 dyn_smem[];
  S* smem = reinterpret_cast<S*>(dyn_smem);
  if (T.rank() == 0) *P.info = 0;
  if (P.n <= 0) return;
  T.stamp(0);
  if (!prepare(T, P)) return;
  if (!cholesky(T, P, smem)) return;
  T.stamp(1);
  if (!reduce_standard(T, P)) return;
  T.stamp(2);
  if (!tridiagonalise(T, P, smem)) return;
  T.stamp(3);
  if (!tridiagonal_eig(T, P, smem)) return;
  T.stamp(5);
  if (!back_transform(T, P, P.smem_cols ? smem : nullptr)) return;
  finish(T, P);
  T.stamp(6);
}

template <class S>
__global__ void __launch_bounds__(kThreads, 1) hegv_grid_kernel(Pencil<S> P, Ctl* ctl, unsigned long long limit_ns) {
  GridTeam T{ctl, P.info, limit_ns};
  solve_pencil(T, P);
}

template <class S>
__global__ void __launch_bounds__(kThreads, 2) hegv_cta_kernel(const Pencil<S>* __restrict__ items, int count) {
  if ((int)blockIdx.x >= count) return;
  const Pencil<S> P = items[blockIdx.x];
  CtaTeam T;
  solve_pencil(T, P);
}

template <class S>
__global__ void __launch_bounds__(kThreads, 2) hegv_cluster_kernel(const Pencil<S>* __restrict__ items, int csize) {
  const Pencil<S> P = items[blockIdx.x / csize];
  ClusterTeam T{(int)blockIdx.x % csize, csize};
  solve_pencil(T, P);
}

size_t pad32(size_t x) { return (x + 31) & ~(size_t)31; }

// Workspace doubles of one pencil, each array padded to 32 doubles: complex, R (complex n^2);
// real, the compact A, B and R (n^2 each); then Z (n^2), wk (6 n^2) and vec (11 n + 8).
size_t work_doubles(int n, bool real) {
  const size_t nn = (size_t)n * n;
  const size_t own = real ? 3 * pad32(nn) : pad32(2 * nn);
  return own + pad32(nn) + pad32(6 * nn) + pad32(11 * (size_t)n + 8);
}

template <class S>
Pencil<S> make_pencil(double2* A, int lda, double2* B, int ldb, double* w, int* info, int n, double* ws) {
  const size_t nn = (size_t)n * n;
  Pencil<S> P;
  P.w = w;
  P.info = info;
  P.n = n;
  P.outA = A;
  P.outB = B;
  P.ldoa = lda;
  P.ldob = ldb;
  double* rest;
  if constexpr (sizeof(S) == sizeof(double)) {  // real: compact copies in the workspace
    P.A = reinterpret_cast<S*>(ws);
    P.B = reinterpret_cast<S*>(ws + pad32(nn));
    P.R = reinterpret_cast<S*>(ws + 2 * pad32(nn));
    P.lda = P.ldb = n;
    rest = ws + 3 * pad32(nn);
  } else {
    P.A = reinterpret_cast<S*>(A);
    P.B = reinterpret_cast<S*>(B);
    P.lda = lda;
    P.ldb = ldb;
    P.R = reinterpret_cast<S*>(ws);
    rest = ws + pad32(2 * nn);
  }
  P.Z = rest;
  P.wk = P.Z + pad32(nn);
  P.vec = P.wk + pad32(6 * nn);
  P.smem_cols = 0;
  P.resident = 0;
  return P;
}

constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s per grid-barrier wait
constexpr int kGridMinN = 32;  // a single pencil at least this large runs on a cooperative grid

// Dynamic shared memory: 3 n words of S for the tridiagonalisation's v_j, w and v_{j+1}, and, when
// it fits in 200 KB, one column of n words of S per warp for the back-transformation.
size_t col_smem_bytes(int n, size_t ws) {
  const size_t b = (size_t)kWarps * (size_t)std::max(n, 1) * ws;
  return b <= 200u * 1024u ? b : 0;
}
size_t dyn_smem_bytes(int n, size_t ws) {
  const size_t chol = ws == 8 ? chol_smem<double>() : chol_smem<double2>();
  return std::max({col_smem_bytes(n, ws), (size_t)3 * std::max(n, 1) * ws, chol});
}
// The tridiagonalisation's vectors and the columns of a CTA of a team of `ctas`, 0 when above `limit`.
size_t resident_smem_bytes(int n, size_t ws, int ctas, size_t limit) {
  const size_t b = ws * (size_t)std::max(n, 1) * (3 + (std::max(n, 1) + ctas - 1) / ctas);
  return b <= limit ? b : 0;
}
constexpr int kMaxN = 4608;  // 3 n complex words must fit in shared memory (221 KB)

// Shared memory of one CTA of a batch on teams of `ctas`; resident: with its columns.  Two CTAs share an
// SM (their registers), so the columns may take half of its shared memory.
size_t batch_smem(int n, size_t ws, int ctas, bool* resident = nullptr) {
  const size_t res = resident_smem_bytes(n, ws, ctas, 110u * 1024u);
  if (resident) *resident = res != 0;
  return std::max(dyn_smem_bytes(n, ws), res);
}

// CTAs per pencil of a batch (orders n[], words of ws bytes), a portable cluster at most and four columns
// a CTA at least: the size with the shortest estimated time, in units of the largest pencil on one CTA.
//   * c CTAs take t = s + (1 - s) / c, the serial share s being 10 / n complex and 18 / n real;
//   * two CTAs on an SM slow each other by the share b = (1 - s) / c / t of their time that is not serial:
//     f = 1 + 0.7 b^1.5;
//   * a wave is two CTAs an SM, less 4 and 5 % for clusters of 4 and 8, which do not span the chip's SM groups; a
//     last wave of half that or less has its SMs to itself;
//   * pencils of uneven order count by their order cubed (the large ones start first).
// Fitted to batches of 20 to 1000 equal pencils of orders 20 to 260 on 1, 2, 4 and 8 CTAs each: within 0.6 %
// of the best size on average, 8 % at most.  (As many CTAs as six an SM allow took up to 1.7 times the
// best for 76 or 152 pencils, more than one CTA each had taken: 152 of order 64 complex 5.95 -> 3.98 ms, of
// order 150 35.5 -> 26.7; 217 uneven ones of 20 to 141, on 1, 2, 4, 8 CTAs 28.0, 18.5, 14.5, 18.2 ms, stay
// on 4.)
template <class P>
int cluster_size(kss_ctx ctx, const std::vector<P>& pencils, int nmax, size_t ws) {
  const double s = std::min(0.7, (ws == 8 ? 18.0 : 10.0) / nmax), nsm = std::max(ctx->nsm, 1);
  double count = 0;
  for (const auto& p : pencils) count += std::pow((double)p.n / nmax, 3);
  if (count > 0.8 * pencils.size()) count = (double)pencils.size();
  int best = 1;
  double tbest = 1e300;
  for (int c = 8; c >= 1; c /= 2) {
    if (c > 1 && 4 * c > nmax) continue;
    const bool pairs = batch_smem(nmax, ws, c) <= 113u * 1024u;
    const double t = s + (1.0 - s) / c, b = (1.0 - s) / c / t, f = pairs ? 1.0 + 0.7 * std::pow(b, 1.5) : 1.0;
    const double wave = (pairs ? 2 : 1) * nsm / c * (c == 8 ? 0.95 : c == 4 ? 0.96 : 1.0);
    const double full = std::floor(count / wave), rest = count - full * wave;
    const double time = t * (full * f + (rest < 1e-9 ? 0.0 : 2.0 * rest <= wave + 4.0 ? 1.0 : f));
    if (time < tbest) {
      tbest = time;
      best = c;
    }
  }
  return best;
}

template <class S>
void launch_cta(kss_ctx ctx, std::vector<Pencil<S>>& small, size_t items_offset, const char* name) {
  if (small.empty()) return;
  // largest pencils first: the CTAs start in launch order, so the long solves begin on their own
  // SMs and the short ones fill in behind them (each CTA reads its own self-contained item)
  std::stable_sort(small.begin(), small.end(), [](const Pencil<S>& a, const Pencil<S>& b) { return a.n > b.n; });
  cudaStream_t st = ctx->stream;
  int nmax = 1;
  for (const auto& P : small) nmax = std::max(nmax, P.n);
  const int csize = cluster_size(ctx, small, nmax, sizeof(S));
  bool res = false;
  const size_t sm = batch_smem(nmax, sizeof(S), csize, &res);
  for (auto& P : small) {
    P.smem_cols = col_smem_bytes(nmax, sizeof(S)) ? 1 : 0;
    P.resident = res ? 1 : 0;
  }
  Pencil<S>* d_items = reinterpret_cast<Pencil<S>*>(static_cast<char*>(ctx->dense_items.p) + items_offset);
  KSS_CHECK_CUDA(cudaMemcpyAsync(d_items, small.data(), small.size() * sizeof(Pencil<S>), cudaMemcpyHostToDevice, st));
  ProfScope ps(ctx, prof_register(name));
  if (csize == 1) {
    KSS_CHECK_CUDA(cudaFuncSetAttribute(hegv_cta_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    hegv_cta_kernel<S><<<(unsigned)small.size(), kThreads, sm, st>>>(d_items, (int)small.size());
  } else {
    KSS_CHECK_CUDA(cudaFuncSetAttribute(hegv_cluster_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)csize;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(small.size() * csize));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    KSS_CHECK_CUDA(cudaLaunchKernelEx(&cfg, hegv_cluster_kernel<S>, (const Pencil<S>*)d_items, csize));
  }
  KSS_CHECK_CUDA(cudaGetLastError());
}

template <class S>
void launch_grid(kss_ctx ctx, Pencil<S> P, const char* name) {
  cudaStream_t st = ctx->stream;
  const int n = P.n;
  const int want = std::max(1, std::min((n + 3) / 4, ctx->nsm > 0 ? ctx->nsm : 1));
  const size_t res = resident_smem_bytes(n, sizeof(S), want, 220u * 1024u);
  const size_t sm = std::max(dyn_smem_bytes(n, sizeof(S)), res);
  KSS_CHECK_CUDA(cudaFuncSetAttribute(hegv_grid_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  int per_sm = 0;
  KSS_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hegv_grid_kernel<S>, kThreads, sm));
  const int coop = std::max(1, per_sm) * std::max(1, ctx->nsm);
  const int G = std::min(want, coop);
  P.resident = res && G == want ? 1 : 0;
  ctx->dense_ctl.ensure(sizeof(Ctl));
  KSS_CHECK_CUDA(cudaMemsetAsync(ctx->dense_ctl.p, 0, sizeof(Ctl), st));
  P.smem_cols = col_smem_bytes(n, sizeof(S)) ? 1 : 0;
  Ctl* ctl = ctx->dense_ctl.as<Ctl>();
  unsigned long long lim = kWaitLimitNs;
  void* args[] = {&P, &ctl, &lim};
  ProfScope ps(ctx, prof_register(name));
  KSS_CHECK_CUDA(cudaLaunchCooperativeKernel((const void*)hegv_grid_kernel<S>, dim3(G), dim3(kThreads), args, sm, st));
}

}  // namespace

void hegv_batched(kss_ctx ctx, const std::vector<HegvItem>& items) {
  if (items.empty()) return;
  size_t total = 0;
  for (const auto& it : items) total += work_doubles(std::max(it.n, 1), it.real);
  ctx->dense_ws.ensure(total * sizeof(double));
  // a CTA or a cluster of them per pencil, real and complex pencils in separate launches; a single large
  // pencil on a cooperative grid
  std::vector<Pencil<double>> small_r;
  std::vector<Pencil<double2>> small_c;
  double* p = ctx->dense_ws.as<double>();
  const bool alone = items.size() == 1;
  for (const auto& it : items) {
    KSS_REQUIRE(it.n >= 0 && it.lda >= std::max(it.n, 1) && it.ldb >= std::max(it.n, 1), "hegv: bad sizes");
    KSS_REQUIRE(it.n <= kMaxN, "hegv: order above " + std::to_string(kMaxN));
    double2* A = (double2*)it.A;
    double2* B = (double2*)it.B;
    const bool large = alone && it.n >= kGridMinN;
    if (it.real) {
      const Pencil<double> P = make_pencil<double>(A, it.lda, B, it.ldb, it.w, it.info, it.n, p);
      if (large) launch_grid(ctx, P, "dense_hegv_grid_real");
      else small_r.push_back(P);
    } else {
      const Pencil<double2> P = make_pencil<double2>(A, it.lda, B, it.ldb, it.w, it.info, it.n, p);
      if (large) launch_grid(ctx, P, "dense_hegv_grid");
      else small_c.push_back(P);
    }
    p += work_doubles(std::max(it.n, 1), it.real);
  }
  const size_t off_c = (small_r.size() * sizeof(Pencil<double>) + 255) & ~(size_t)255;
  ctx->dense_items.ensure(off_c + small_c.size() * sizeof(Pencil<double2>) + 1);
  launch_cta(ctx, small_r, 0, "dense_hegv_cta_real");
  launch_cta(ctx, small_c, off_c, "dense_hegv_cta");
}

void hegv(kss_ctx ctx, int n, void* A, int lda, void* B, int ldb, double* w, int* info, bool real) {
  hegv_batched(ctx, {HegvItem{A, B, w, info, n, lda, ldb, real}});
}

}  // namespace kss

using namespace kss;

extern "C" kss_status kss_dense_hegv(kss_ctx ctx, int count, const int* n, void* const* A, const int* lda,
                                     void* const* B, const int* ldb, double* const* w, int* info, int real) {
  if (!ctx) return KSS_EINVAL;
  try {
    KSS_REQUIRE(count >= 0, "count < 0");
    if (count == 0) {
      ctx->err.clear();
      return KSS_OK;
    }
    KSS_REQUIRE(n && A && lda && B && ldb && w && info, "NULL argument");
    KSS_CHECK_CUDA(cudaSetDevice(ctx->device));
    std::vector<HegvItem> items(count);
    DevBuf dinfo;
    dinfo.alloc((size_t)count * sizeof(int));
    for (int i = 0; i < count; ++i) {
      KSS_REQUIRE(n[i] >= 0 && lda[i] >= std::max(1, n[i]) && ldb[i] >= std::max(1, n[i]), "bad order or leading dimension");
      KSS_REQUIRE(n[i] == 0 || (A[i] && B[i] && w[i]), "NULL matrix");
      items[i] = HegvItem{A[i], B[i], w[i], dinfo.as<int>() + i, n[i], lda[i], ldb[i], real != 0};
    }
    hegv_batched(ctx, items);
    KSS_CHECK_CUDA(cudaMemcpyAsync(info, dinfo.p, (size_t)count * sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    KSS_CHECK_CUDA(cudaStreamSynchronize(ctx->stream));
    KSS_CHECK_CUDA(cudaGetLastError());
    for (int i = 0; i < count; ++i)
      if (info[i] < 0) fail(KSS_ETIMEOUT, "kss_dense_hegv: a bounded grid-barrier wait gave up");
    ctx->err.clear();
    return KSS_OK;
  } catch (const KssError& e) {
    ctx->err = e.msg;
    return e.st;
  } catch (...) {
    ctx->err = "unexpected internal error";
    return KSS_ECUDA;
  }
}

extern "C" kss_status kss_dense_hegv_phase_ms(kss_ctx ctx, double* ms) {
  if (!ctx || !ms) return KSS_EINVAL;
  try {
    for (int k = 0; k < 6; ++k) ms[k] = 0.0;
    if (!ctx->dense_ctl.p) {
      ctx->err.clear();
      return KSS_OK;
    }
    KSS_CHECK_CUDA(cudaSetDevice(ctx->device));
    Ctl c;
    KSS_CHECK_CUDA(cudaMemcpyAsync(&c, ctx->dense_ctl.p, sizeof(Ctl), cudaMemcpyDeviceToHost, ctx->stream));
    KSS_CHECK_CUDA(cudaStreamSynchronize(ctx->stream));
    if (c.t[6] > c.t[0])
      for (int k = 0; k < 6; ++k) ms[k] = c.t[k + 1] > c.t[k] ? 1e-6 * (double)(c.t[k + 1] - c.t[k]) : 0.0;
    ctx->err.clear();
    return KSS_OK;
  } catch (const KssError& e) {
    ctx->err = e.msg;
    return e.st;
  }
}

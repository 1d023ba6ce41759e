// Small complex128 products on the FP64 pipe: C = alpha A^H B + beta C with a long K (projector
// coefficients, Gram matrices) and C = alpha A B + beta C with a long M (nonlocal accumulation,
// rotations) of blocks of a few dozen bands, where the digit products of gemm_oz.cu spend their time
// on operand preparation, pipeline fill and drains that the size does not repay.
//
// What bounds them: FP64 issue.  A warp's FP64 instruction holds its quarter of the SM for 64 cycles, so
// the work is spread thinly: one output per thread (16 x 8 outputs per CTA, K split until every SM
// has two CTAs; 32 x 4 outputs per CTA in the product without a split), operands through shared memory
// or L1, four fused multiply-adds per term.  The K splits are added in a fixed order.
//
// Measured: H on 20 bands of a cell with 16 projectors and 1503 plane waves 195 -> 96 us, a solve of
// it 65 -> 25 ms.  Error of a product with 9200 terms 2e-15 of its largest entry (digits: 1.4e-14).
#include <algorithm>
#include <string>

#include "kss_internal.h"

namespace kss {

namespace {

constexpr int kT = 128;
constexpr int BM = 16, BN = 8, BK = 16;  // product with K split: outputs and K step of a CTA
constexpr int RM = 32, RN = 4;           // product without: outputs of a CTA

__global__ void __launch_bounds__(kT) small_cn_partial(int M, int N, int K, const double2* __restrict__ A, long long lda,
                                                       const double2* __restrict__ B, long long ldb,
                                                       double2* __restrict__ P, int tm, int tn, int kchunk) {
  __shared__ double2 As[BK][BM + 1], Bs[BK][BN + 1];
  const int tid = threadIdx.x;
  const int t = blockIdx.x, z = t / (tm * tn), r = t - z * (tm * tn);
  const int i0 = (r % tm) * BM, j0 = (r / tm) * BN;
  const int k0 = z * kchunk, k1 = min(K, k0 + kchunk);
  const int lk = tid & (BK - 1), l = tid / BK;  // k fastest: 256-byte rows
  const int i = tid & (BM - 1), j = tid / BM;
  double2 a[2], b;
  auto fetch = [&](int k) {
    const bool in = k + lk < k1;
    const double2 zero = make_double2(0, 0);
    a[0] = in && i0 + l < M ? A[(i0 + l) * lda + k + lk] : zero;
    a[1] = in && i0 + l + 8 < M ? A[(i0 + l + 8) * lda + k + lk] : zero;
    b = in && j0 + l < N ? B[(j0 + l) * ldb + k + lk] : zero;
  };
  double2 acc = make_double2(0, 0);
  fetch(k0);
  for (int k = k0; k < k1; k += BK) {
    As[lk][l] = a[0];
    As[lk][l + 8] = a[1];
    Bs[lk][l] = b;
    __syncthreads();
    if (k + BK < k1) fetch(k + BK);
#pragma unroll
    for (int q = 0; q < BK; ++q) {
      const double2 x = As[q][i], y = Bs[q][j];
      acc.x = fma(x.y, y.y, fma(x.x, y.x, acc.x));
      acc.y = fma(-x.y, y.x, fma(x.x, y.y, acc.y));
    }
    __syncthreads();
  }
  if (i0 + i < M && j0 + j < N) P[(size_t)z * M * N + (size_t)(j0 + j) * M + i0 + i] = acc;
}

__device__ __forceinline__ void store(double2* dst, double2 v, double ar, double ai, double br, double bi) {
  if (ar != 1.0 || ai != 0.0) v = make_double2(ar * v.x - ai * v.y, ar * v.y + ai * v.x);
  if (br != 0.0 || bi != 0.0) {
    const double2 o = *dst;
    if (br == 1.0 && bi == 0.0) v = make_double2(v.x + o.x, v.y + o.y);
    else v = make_double2(v.x + (br * o.x - bi * o.y), v.y + (br * o.y + bi * o.x));
  }
  *dst = v;
}

// Sum of the splits, eight lanes an output; rows scaled by rs[i] s when rs is given.
__global__ void __launch_bounds__(kT) small_cn_reduce(int M, int N, int splits, const double2* __restrict__ P,
                                                      const double* __restrict__ rs, double s, double2* __restrict__ C,
                                                      long long ldc, double ar, double ai, double br, double bi) {
  const long long o = blockIdx.x * (long long)(kT / 8) + threadIdx.x / 8;
  const int q = threadIdx.x & 7;
  const size_t mn = (size_t)M * N;
  double2 v = make_double2(0, 0);
  if (o < (long long)mn) {
#pragma unroll 4
    for (int z = q; z < splits; z += 8) {
      const double2 p = P[z * mn + o];
      v.x += p.x;
      v.y += p.y;
    }
  }
#pragma unroll
  for (int w = 4; w > 0; w >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, w);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, w);
  }
  if (q || o >= (long long)mn) return;
  const int i = (int)(o % M);
  if (rs) {
    const double f = rs[i] * s;
    v.x *= f;
    v.y *= f;
  }
  store(C + (o / M) * ldc + i, v, ar, ai, br, bi);
}

__global__ void __launch_bounds__(kT) small_nn(int M, int N, int K, const double2* __restrict__ A, long long lda,
                                               const double2* __restrict__ B, long long ldb, double2* __restrict__ C,
                                               long long ldc, int tm, double ar, double ai, double br, double bi) {
  const int i = (blockIdx.x % tm) * RM + (threadIdx.x & 31), j = (blockIdx.x / tm) * RN + (threadIdx.x >> 5);
  if (i >= M || j >= N) return;
  const double2* __restrict__ pa = A + i;
  const double2* __restrict__ pb = B + j * ldb;
  double2 acc = make_double2(0, 0);
#pragma unroll 8
  for (int k = 0; k < K; ++k) {
    const double2 x = pa[k * lda], y = pb[k];  // pb: one address per warp
    acc.x = fma(-x.y, y.y, fma(x.x, y.x, acc.x));
    acc.y = fma(x.y, y.x, fma(x.x, y.y, acc.y));
  }
  store(C + j * ldc + i, acc, ar, ai, br, bi);
}

}  // namespace

// Up to this many terms the FP64 pipe is faster than the digit products, whose time hardly depends on the
// size there (kss_gemm, us, digit products / here; coefficients: 0.5M terms 122 / 25, 7.7M 129 / 77,
// 15.8M 129 / 152; accumulation: 0.5M 61 / 41, 7.7M 75 / 90).
// The sum over the splits takes eight lanes an output (at 65536 outputs 10 us), and the form without a
// split one thread (at 256 terms 35 us).
bool small_product_cn(int M, int N, int K) { return (double)M * N * K <= 12e6 && (double)M * N <= 65536; }
bool small_product_nn(int M, int N, int K) { return (double)M * N * K <= 4e6 && K <= 256; }

void small_gemm_cn(kss_ctx ctx, int M, int N, int K, const void* A, int lda, const void* B, int ldb, void* C, int ldc,
                   double ar, double ai, double br, double bi, const char* tag, const double* row_scale, double s) {
  if (M <= 0 || N <= 0) return;
  const long long tm = (M + BM - 1) / BM, tn = (N + BN - 1) / BN;
  const int nsm = std::max(ctx->nsm, 1);
  const long long want = std::max(1LL, std::min<long long>(2LL * nsm / (tm * tn), (K + BK - 1) / BK));
  const int kchunk = (int)(((K + want - 1) / want + BK - 1) / BK * BK);
  const int splits = (K + kchunk - 1) / kchunk;
  ctx->oz_part.ensure((size_t)splits * M * N * sizeof(double2));
  double2* P = ctx->oz_part.as<double2>();
  {
    ProfScope ps(ctx, prof_register((std::string("gemm64_small:") + tag).c_str()));
    small_cn_partial<<<(unsigned)(tm * tn * splits), kT, 0, ctx->stream>>>(M, N, K, (const double2*)A, lda,
                                                                           (const double2*)B, ldb, P, (int)tm, (int)tn,
                                                                           kchunk);
  }
  {
    ProfScope ps(ctx, prof_register((std::string("gemm64_small_reduce:") + tag).c_str()));
    const long long mn = (long long)M * N;
    small_cn_reduce<<<(unsigned)((mn + kT / 8 - 1) / (kT / 8)), kT, 0, ctx->stream>>>(M, N, splits, P, row_scale, s,
                                                                                      (double2*)C, ldc, ar, ai, br, bi);
  }
  KSS_CHECK_CUDA(cudaGetLastError());
}

void small_gemm_nn(kss_ctx ctx, int M, int N, int K, const void* A, int lda, const void* B, int ldb, void* C, int ldc,
                   double ar, double ai, double br, double bi, const char* tag) {
  if (M <= 0 || N <= 0) return;
  const long long tm = (M + RM - 1) / RM, tn = (N + RN - 1) / RN;
  ProfScope ps(ctx, prof_register((std::string("gemm64_small:") + tag).c_str()));
  small_nn<<<(unsigned)(tm * tn), kT, 0, ctx->stream>>>(M, N, K, (const double2*)A, lda, (const double2*)B, ldb,
                                                        (double2*)C, ldc, (int)tm, ar, ai, br, bi);
  KSS_CHECK_CUDA(cudaGetLastError());
}

}  // namespace kss

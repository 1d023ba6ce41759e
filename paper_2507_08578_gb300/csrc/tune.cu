// Autotuner of the FFT radix schedule of pass B (the y/z transforms of the local-potential path,
// §5.1 batched FFTs).  For a box length N = N2 = N3 the candidates are the CTA-wide form with
// every compile-time split N = A * B at 256 and 384 threads per CTA (and 128 in single precision),
// in fixed point where the caller runs it so (double precision), and the per-warp form.  Each
// candidate runs one warm-up and three timed launches (the fastest counts) on a scratch slab of
// the same window and of the production chunk size (CUDA events on the context's stream): zeros in
// floating point, whose time does not depend on the values, and values of the size that pass A leaves
// in fixed point; the fastest candidate is kept for the process in a table keyed by device, precision,
// box and window.  All candidates compute the same transform; they differ only in rounding order.
#include <map>
#include <mutex>
#include <tuple>

#include "gemm_tune.h"
#include "local_wide.h"
#include "tune.h"

namespace kss {

namespace {

using Key = std::tuple<int, int, int, int, int, int>;  // device, bytes/real, N1, N2, N3, W3 (rounded)

struct Entry {
  PassBSched s;
  int device, prec, N1, N, W3, W2;
};

// What is kept for a configuration: a schedule of the floating-point passes and one of the
// fixed-point passes (double precision).  The table has one entry for both, the fixed-point one where
// that is there, and a pinned schedule is pinned for both.
struct Slot {
  Entry e[2];
  bool has[2] = {false, false};
};

std::mutex g_mu;
std::map<Key, Slot> g_table;
std::vector<Key> g_order;  // insertion order (for listing)

// The CTA-wide pass B of schedule c, in fixed point (fx) or in the data's precision (dry: whether there is one).
template <typename T>
bool wide(const lk::LocalArgs<T>& a, const PassBSched& c, bool fx, int nbands, cudaStream_t st, bool dry) {
  if constexpr (sizeof(T) == 8) {
    if (fx) return fx_pass_b(a, c.A, c.B, c.threads, nbands, st, dry);
  }
  return wide_pass_b<T>(a, c.A, c.B, c.threads, nbands, st, dry);
}

// A fixed-point slab like those of pass A, with the plane entries to match, and V as the pass reads it (its
// layout aside).  On zeros the pass would shift a plane before six of its eight stages (measured on a
// slab of zeros: 2 to 5 % above the same launch on bands, more for some splits than for others).
__global__ void fill_fx(long long* work, long long n, int2* ma, long long nm, fx::Limbs* V, long long nv,
                        const double* __restrict__ Vx, double points, const int* __restrict__ vhigh) {
  const int E = fx::v_exp(*vhigh) - 63;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n || i < nv;
       i += (long long)gridDim.x * blockDim.x) {
    if (i < n) work[i] = fx::slab_value((unsigned long long)i);
    if (i < nm) ma[i] = make_int2(0, fx::kSlabBits);
    if (i < nv) V[i] = fx::limbs(fx::from_double(Vx[i] * points, E));
  }
}

template <typename T>
PassBSched builtin(const lk::LocalArgs<T>& a, const fftr::Split& s2, bool fx) {
  PassBSched s{s2.A, s2.B, lk::kWideThreads, 0, 0};
  if (!wide(a, s, fx, 0, nullptr, true)) s.threads = 0;
  return s;
}

}  // namespace

template <typename T>
PassBSched pass_b_schedule(kss_ctx ctx, const lk::LocalArgs<T>& a, const fftr::Split& s2, bool may_tune, bool fx) {
  // Configurations are keyed by box and the window height W3 rounded up to a multiple of 8 (the
  // y-stage task count).  A candidate has to fit at the rounded height, so that the choice fits every
  // smaller one; it is timed on the caller's own window, which decides between the pruned and the full
  // instance of a split.
  const int W3b = std::min(a.N3, (a.W3 + 7) / 8 * 8);
  const Key key{ctx->device, (int)sizeof(T), a.N1, a.N2, a.N3, W3b};
  {
    std::lock_guard<std::mutex> lock(g_mu);
    auto it = g_table.find(key);
    if (it != g_table.end() && it->second.has[fx]) return it->second.e[fx].s;
  }
  if (!may_tune || !ctx->autotune) return builtin<T>(a, s2, fx);
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  KSS_CHECK_CUDA(cudaStreamIsCapturing(ctx->stream, &cs));
  if (cs != cudaStreamCaptureStatusNone) return builtin<T>(a, s2, fx);

  KSS_REQUIRE(!fx || (a.fx.r2 && a.fx.vhigh), "pass-B tuner: arguments without the fixed-point tables");

  using C = typename lk::CT<T>::C;
  lk::LocalArgs<T> t = a, tall = a;
  tall.W3 = W3b;
  // candidates: CTA-wide splits x threads, then the per-warp form
  std::vector<PassBSched> cand;
  if (a.N2 == a.N3)
    for (const auto& ab : wide_splits())
      for (int nt : {128, 256, 384}) {  // 128: single precision only (the dry check says which exist)
        const PassBSched c{ab.first, ab.second, nt, 0, 0};
        if (c.A * c.B == a.N2 && wide(tall, c, fx, 0, nullptr, true)) cand.push_back(c);
      }
  cand.push_back(PassBSched{s2.A, s2.B, 0, 0, 0});
  // scratch slab of the production chunk size (the local passes keep kSlabChunkBytes of slab per
  // launch), so that candidates are timed at the launch shape they will run at
  const size_t per_band = (size_t)t.N1 * t.W3 * t.W2 * sizeof(C);
  const int nbt = (int)std::max<size_t>(1, std::min<size_t>(64, kSlabChunkBytes / per_band));
  const size_t elems = (size_t)t.N1 * t.W3 * t.W2 * nbt;
  const size_t nmeta = (size_t)nbt * (t.N1 + t.W3), nv = fx ? (size_t)t.N1 * t.N2 * t.N3 : 0;
  const size_t bytes = elems * sizeof(C) + (fx ? sizeof(int2) * nmeta + sizeof(fx::Limbs) * nv : 0);
  ctx->ws_tune.ensure(bytes);
  t.work = ctx->ws_tune.as<C>();
  // (a launch overwrites the slab, whose plane entries then no longer hold: filled anew for each)
  auto refill = [&](const PassBSched& c) {
    if constexpr (sizeof(T) == 8) {
      if (fx && c.threads) {
        t.fx.ma = reinterpret_cast<int2*>(t.work + elems);
        t.fx.mb = t.fx.ma + (size_t)nbt * t.W3;
        fx::Limbs* V = reinterpret_cast<fx::Limbs*>(t.fx.ma + nmeta);
        t.fx.V = V;
        fill_fx<<<152 * 8, 256, 0, ctx->stream>>>(reinterpret_cast<long long*>(t.work), 2 * (long long)elems, t.fx.ma,
                                                  (long long)nmeta, V, (long long)nv, t.Vx,
                                                  (double)t.N1 * t.N2 * t.N3, t.fx.vhigh);
        KSS_CHECK_CUDA(cudaGetLastError());
        return;
      }
    }
    KSS_CHECK_CUDA(cudaMemsetAsync(ctx->ws_tune.p, 0, elems * sizeof(C), ctx->stream));
  };
  t.Vpi = t.Vx;  // any N1 x N x N array: the values do not matter for timing
  t.n0 = 0;
  cudaEvent_t e0, e1;
  KSS_CHECK_CUDA(cudaEventCreate(&e0));
  KSS_CHECK_CUDA(cudaEventCreate(&e1));
  auto launch = [&](const PassBSched& c) {
    if (c.threads) wide(t, c, fx, nbt, ctx->stream, false);
    else warp_pass_b<T>(ctx, t, nbt);
  };
  int best = -1;
  for (size_t i = 0; i < cand.size(); ++i) {
    refill(cand[i]);
    launch(cand[i]);  // warm-up (and shared-memory attribute)
    double tmin = 1e300;
    for (int r = 0; r < 3; ++r) {  // the fastest of three timed launches
      if (fx) refill(cand[i]);
      KSS_CHECK_CUDA(cudaEventRecord(e0, ctx->stream));
      launch(cand[i]);
      KSS_CHECK_CUDA(cudaEventRecord(e1, ctx->stream));
      KSS_CHECK_CUDA(cudaEventSynchronize(e1));
      float ms = 0;
      KSS_CHECK_CUDA(cudaEventElapsedTime(&ms, e0, e1));
      tmin = std::min(tmin, (double)ms);
    }
    cand[i].ms = tmin;
    if (best < 0 || cand[i].ms < cand[best].ms) best = (int)i;
  }
  KSS_CHECK_CUDA(cudaEventDestroy(e0));
  KSS_CHECK_CUDA(cudaEventDestroy(e1));
  KSS_CHECK_CUDA(cudaGetLastError());
  PassBSched s = cand[best];
  s.ncand = (int)cand.size();
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_table.count(key)) g_order.push_back(key);
  Slot& slot = g_table[key];
  if (!slot.has[fx]) {
    slot.e[fx] = Entry{s, ctx->device, sizeof(T) == 8 ? KSS_PREC_FP64 : KSS_PREC_MIXED, a.N1, a.N2, W3b, a.W2};
    slot.has[fx] = true;
  }
  return slot.e[fx].s;
}

template PassBSched pass_b_schedule<double>(kss_ctx, const lk::LocalArgs<double>&, const fftr::Split&, bool, bool);
template PassBSched pass_b_schedule<float>(kss_ctx, const lk::LocalArgs<float>&, const fftr::Split&, bool, bool);

}  // namespace kss

using namespace kss;

extern "C" {

kss_status kss_autotune_set(kss_ctx ctx, int mode) {
  if (!ctx || (mode != 0 && mode != 1)) return KSS_EINVAL;
  ctx->autotune = mode;
  return KSS_OK;
}

kss_status kss_autotune_count(int* n) {
  if (!n) return KSS_EINVAL;
  std::lock_guard<std::mutex> lock(g_mu);
  *n = (int)g_order.size();
  return KSS_OK;
}

kss_status kss_autotune_get(int i, kss_tune_entry* out) {
  if (!out) return KSS_EINVAL;
  std::lock_guard<std::mutex> lock(g_mu);
  if (i < 0 || i >= (int)g_order.size()) return KSS_EINVAL;
  const Slot& slot = g_table.at(g_order[i]);
  const Entry& e = slot.e[slot.has[1]];
  out->device = e.device;
  out->precision = e.prec;
  out->N1 = e.N1;
  out->N = e.N;
  out->W3 = e.W3;
  out->W2 = e.W2;
  out->A = e.s.A;
  out->B = e.s.B;
  out->threads = e.s.threads;
  out->ms = e.s.ms;
  out->ncand = e.s.ncand;
  return KSS_OK;
}

kss_status kss_autotune_put(const kss_tune_entry* e) {
  if (!e || e->N1 < 2 || e->N < 2 || e->W3 < 1 || e->W3 > e->N ||
      (e->precision != KSS_PREC_FP64 && e->precision != KSS_PREC_MIXED) ||
      (e->threads != 0 && e->threads != 128 && e->threads != 256 && e->threads != 384) || e->A * e->B != e->N)
    return KSS_EINVAL;
  const int bytes = e->precision == KSS_PREC_FP64 ? 8 : 4;
  const int W3b = std::min(e->N, (e->W3 + 7) / 8 * 8);
  const Key key{e->device, bytes, e->N1, e->N, e->N, W3b};
  PassBSched s;
  s.A = e->A;
  s.B = e->B;
  s.threads = e->threads;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_table.count(key)) g_order.push_back(key);
  Slot& slot = g_table[key];
  slot.e[0] = slot.e[1] = Entry{s, e->device, e->precision, e->N1, e->N, W3b, e->W2};
  slot.has[0] = slot.has[1] = true;
  return KSS_OK;
}

kss_status kss_autotune_clear(void) {
  {
    std::lock_guard<std::mutex> lock(g_mu);
    g_table.clear();
    g_order.clear();
  }
  gemm_tune_clear();
  return KSS_OK;
}

}  // extern "C"

// Plan autotuner: picks the launch shapes of the kernels that dominate a
// solve by timing the candidates on the plan's own buffers, once per
// (grid, K, right-hand sides, restart, precision) in a process, and caches
// the choice.  Candidates:
//   symbol pass       nodes per block {1, 2, 4} (the spectrum is read once
//                     per block; fewer, longer blocks), one or two columns
//                     per thread (complex64)
//   x-inverse pass    fused weighted sum, or in place + gather
// The Gram-Schmidt kernels have one launch shape; their times are reported.
// Timing uses CUDA events on the caller's stream around 3 repetitions of
// each candidate at the middle Arnoldi step of a cycle.
#include <algorithm>
#include <cstdlib>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "hz_internal.h"
#include "kernels.h"

namespace hz {
hz_status precond_apply(hz_plan* p, int prec, const double2* in, const double* scale, int nrhs,
                        void* out, int out_kind, cudaStream_t st, const int* active,
                        bool by_size = false);
}

using namespace hz;

namespace {

using Key = std::tuple<int, int, int, int, int, int, int>;
std::mutex g_mu;
std::map<Key, Tune> g_cache;

Key key_of(const hz_plan* p) {
  const hz_medium* m = p->med;
  return Key(m->nx, m->ny, m->nz, m->K, p->max_nrhs, p->opts.restart, p->opts.precision);
}

struct Timer {
  cudaEvent_t a = nullptr, b = nullptr;
  cudaStream_t st;
  explicit Timer(cudaStream_t s) : st(s) {
    cudaEventCreate(&a);
    cudaEventCreate(&b);
  }
  ~Timer() {
    cudaEventDestroy(a);
    cudaEventDestroy(b);
  }
  template <typename F>
  float best_ms(F&& f, int reps = 3) {
    float best = 1e30f;
    for (int r = 0; r < reps; ++r) {
      cudaEventRecord(a, st);
      if (f() != HZ_OK) return 1e30f;
      cudaEventRecord(b, st);
      if (cudaEventSynchronize(b) != cudaSuccess) return 1e30f;
      float ms = 0.f;
      cudaEventElapsedTime(&ms, a, b);
      best = std::min(best, ms);
    }
    return best;
  }
};

// the report's fields of the Gram-Schmidt kernels' fixed shape
void gs_shape(hz_tune_report* r) {
  r->dots_bps = 4;
  r->dots_vc = 8;
  r->upd_bps = 4;
}

}  // namespace

// Launch shapes from the process cache without timing: the entry of the
// plan's own key, else the entry of the same grid, K, restart and precision
// whose right-hand-side count is nearest.  The scattering x-inverse is not
// taken for media with per-point (node, weight) records (with three or more
// additions per point its result would depend on their order).
bool hz::tune_from_cache(hz_plan* plan) {
  const Key key = key_of(plan);
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_cache.find(key);
  if (it == g_cache.end()) {
    int best_d = 1 << 30;
    for (auto jt = g_cache.begin(); jt != g_cache.end(); ++jt) {
      const Key& k = jt->first;
      if (std::get<0>(k) != std::get<0>(key) || std::get<1>(k) != std::get<1>(key) ||
          std::get<2>(k) != std::get<2>(key) || std::get<3>(k) != std::get<3>(key) ||
          std::get<5>(k) != std::get<5>(key) || std::get<6>(k) != std::get<6>(key))
        continue;
      const int d = std::abs(std::get<4>(k) - std::get<4>(key));
      if (d < best_d) {
        best_d = d;
        it = jt;
      }
    }
  }
  if (it == g_cache.end()) return false;
  plan->tune = it->second;
  if (plan->med->generic && plan->tune.rowinv_mode == 3) plan->tune.rowinv_mode = 1;
  return true;
}

extern "C" hz_status hz_plan_set_tune(hz_plan* plan, const hz_tune_report* r) {
  if (!plan || !r) return set_error(HZ_ERR_INVALID_ARG, "null argument");
  const bool ok = (r->dots_vc == 2 || r->dots_vc == 4 || r->dots_vc == 8) && r->dots_bps >= 1 &&
                  r->dots_bps <= 4 && r->upd_bps >= 1 && r->upd_bps <= 8 &&
                  (r->syminv_kpb == 1 || r->syminv_kpb == 2 || r->syminv_kpb == 4) &&
                  r->rowinv_mode >= 0 && r->rowinv_mode <= 3 && r->col_pair >= 0 && r->col_pair <= 2;
  if (!ok) return set_error(HZ_ERR_INVALID_ARG, "launch shape out of range");
  plan->tune.syminv_kpb = r->syminv_kpb;
  plan->tune.rowinv_mode = r->rowinv_mode;
  plan->tune.col_pair = r->col_pair;
  plan->tune.by_size = false;
  return HZ_OK;
}

extern "C" hz_status hz_plan_autotune(hz_plan* plan, void* stream, hz_tune_report* rep) {
  if (!plan) return set_error(HZ_ERR_INVALID_ARG, "null plan");
  const Key key = key_of(plan);
  {
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_cache.find(key);
    if (it != g_cache.end()) {
      plan->tune = it->second;
      if (rep) {
        *rep = hz_tune_report{};
        gs_shape(rep);
        rep->syminv_kpb = plan->tune.syminv_kpb;
        rep->rowinv_mode = plan->tune.rowinv_mode;
        rep->col_pair = plan->tune.col_pair;
        rep->cached = 1;
      }
      return HZ_OK;
    }
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  HZ_TRY(solve_ws_create(plan));
  hz_plan* p = plan;
  const hz_medium* med = p->med;
  const long n = med->n;
  const int m = p->opts.restart, B = p->max_nrhs;
  const int j = std::max(0, m / 2);
  const long ldb = B;
  KsDev& ks = p->ws->ks;
  // defined contents for the timed kernels: zero basis, unit scales, all active
  const Basis Q{reinterpret_cast<int4*>(p->V), p->ev, ldb, n, (n + HZ_FX_TILE - 1) / HZ_FX_TILE,
                p->opts.no_precond == 0};
  double2* W = p->V + long(m) * ldb * n;
  HZ_CUDA(cudaMemsetAsync(p->V, 0, size_t(j + 1) * B * n * sizeof(double2), st));
  HZ_CUDA(cudaMemsetAsync(W, 0, size_t(B) * n * sizeof(double2), st));
  HZ_CUDA(cudaMemsetAsync(p->ev, 0, size_t(j + 1) * B * Q.ntiles * sizeof(int), st));
  HZ_CUDA(cudaMemsetAsync(ks.sigma, 0, size_t(m + 1) * B * sizeof(double), st));
  HZ_CUDA(cudaMemsetAsync(ks.S1, 0, size_t(m + 1) * B * sizeof(double2), st));
  std::vector<int> ones(B, 1);
  HZ_CUDA(cudaMemcpyAsync(ks.active, ones.data(), B * sizeof(int), cudaMemcpyHostToDevice, st));
  HZ_CUDA(cudaMemsetAsync(p->tmp, 0, size_t(B) * n * 16, st));
  HZ_CUDA(cudaStreamSynchronize(st));
  Timer tm(st);
  const Tune def;
  Tune best = def;
  hz_tune_report r{};

  // Gram-Schmidt kernels
  r.dots_us = r.dots_us_default = 1e3f * tm.best_ms([&] {
    return launch_dots(Q, W, n, j, B, ks.active, reinterpret_cast<double2*>(p->partial), ks.S1,
                       m + 1, st);
  });
  r.upd_us = r.upd_us_default = 1e3f * tm.best_ms([&] {
    int nblk = 0;
    return launch_update(Q, W, n, j, B, ks.S1, m + 1, ks.sigma, B, ks.active, p->partial, &nblk,
                         false, st);
  });

  // symbol pass, through a whole preconditioner apply (its other passes do
  // not depend on the choice)
  float tbest = 1e30f;
  const int prec = p->opts.precision;
  void* out = p->Z;
  best.by_size = false;
  p->tune = def;  // what an untuned plan's apply does
  const float tdef = tm.best_ms([&] {
    return precond_apply(p, prec, W, nullptr, B, out, prec == 1 ? 0 : 1, st, nullptr, true);
  });
  for (int pair : {1, 2, 0}) {
    if (pair != 1 && prec == 0) continue;  // FP64 has one form
    for (int kpb : {1, 2, 4}) {
      if (kpb > 1 && kpb > med->K) break;
      p->tune = best;
      p->tune.syminv_kpb = kpb;
      p->tune.col_pair = pair;
      const float ms = tm.best_ms([&] {
        return precond_apply(p, prec, W, nullptr, B, out, prec == 1 ? 0 : 1, st, nullptr);
      });
      if (ms < tbest) {
        tbest = ms;
        best.syminv_kpb = kpb;
        best.col_pair = pair;
      }
    }
  }
  // x-inverse pass: fused weighted sum, in place + gather, or one line per
  // (row, node) added into the cleared output.  The last is bitwise
  // reproducible only with at most two additions per point, so it is not a
  // candidate for the four-weight records of the bivariate / quadratic forms.
  for (int mode : {2, 1, 3}) {
    if (mode == 3 && med->generic) continue;
    p->tune = best;
    p->tune.rowinv_mode = mode;
    const float ms = tm.best_ms([&] {
      return precond_apply(p, prec, W, nullptr, B, out, prec == 1 ? 0 : 1, st, nullptr);
    });
    if (ms < tbest) {
      tbest = ms;
      best.rowinv_mode = mode;
    }
  }
  // direct applies keep their shape by size where no candidate beats it (the
  // node loop of sym_shape is not among them)
  best.by_size = tdef <= tbest;
  r.apply_us = 1e3f * std::min(tbest, tdef);
  r.apply_us_default = 1e3f * tdef;
  HZ_CUDA(cudaStreamSynchronize(st));
  p->tune = best;
  gs_shape(&r);
  r.syminv_kpb = best.syminv_kpb;
  r.rowinv_mode = best.rowinv_mode;
  r.col_pair = best.col_pair;
  r.cached = 0;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    g_cache[key] = best;
  }
  if (rep) *rep = r;
  return HZ_OK;
}

// Calls of libkpm on a device whose allocations above a limit fail.  The limit is made
// here, on the host: this program's own cudaMallocAsync and cudaMallocFromPoolAsync come
// before the CUDA runtime's and return cudaErrorMemoryAllocation for larger requests.
// Prints per call: its name, the status without and with the limit, and the largest
// difference of the results.
#include <cuda_runtime_api.h>
#include <dlfcn.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <functional>
#include <vector>

#include "kpm.h"

namespace {
size_t g_limit = SIZE_MAX, g_largest = 0;
bool refused(size_t n) {
  g_largest = std::max(g_largest, n);
  return n > g_limit;
}
}  // namespace

extern "C" cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t s) {
  using F = cudaError_t (*)(void **, size_t, cudaStream_t);
  static F next = reinterpret_cast<F>(dlsym(RTLD_NEXT, "cudaMallocAsync"));
  return refused(n) ? cudaErrorMemoryAllocation : next(p, n, s);
}
extern "C" cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t pool, cudaStream_t s) {
  using F = cudaError_t (*)(void **, size_t, cudaMemPool_t, cudaStream_t);
  static F next = reinterpret_cast<F>(dlsym(RTLD_NEXT, "cudaMallocFromPoolAsync"));
  return refused(n) ? cudaErrorMemoryAllocation : next(p, n, pool, s);
}

namespace {

using Call = std::function<int(std::vector<double> &)>;

// limit: 0 for one byte less than the largest request of the call without a limit
void check(const char *name, const Call &call, size_t limit = 0) {
  std::vector<double> ref, got;
  g_limit = SIZE_MAX;
  g_largest = 0;
  const int rc = call(ref);
  g_limit = limit ? limit : g_largest - 1;
  const int rc_limit = call(got);
  g_limit = SIZE_MAX;
  double diff = 0.0, size = 0.0;
  for (size_t i = 0; i < ref.size(); ++i) {
    diff = std::max(diff, std::isfinite(got[i]) ? std::fabs(got[i] - ref[i]) : INFINITY);
    size = std::max(size, std::fabs(ref[i]));
  }
  std::printf("%s %d %d %.3e %s\n", name, rc, rc_limit, diff / size, kpm_last_error());
}

struct Model {
  std::vector<int32_t> bi, bj;
  std::vector<double> J;
  Model(int n, bool own) {
    for (int d = 1; d <= 2; ++d)
      for (int i = 0; i < n; ++i) {
        bi.push_back(i);
        bj.push_back((i + d) % n);
        J.push_back(own ? 1.0 + 0.01 * i + 0.3 * d : 1.0 / d);
      }
  }
  kpm_model of(int n) const { return {n, (int32_t)J.size(), bi.data(), bj.data(), J.data()}; }
};

}  // namespace

int main() {
  for (int own = 0; own < 2; ++own)
    for (int n : {12, 16})
      for (int precision : {KPM_FP64, KPM_FP32}) {
        const Model m(n, own);
        const kpm_model km = m.of(n);
        const int32_t up = n / 2;
        const double a = 30.0, b = 0.0;
        char name[64];
        std::snprintf(name, sizeof(name), "moments-%d-%d-%d", own, n, precision);
        check(name, [&](std::vector<double> &mu) {
          mu.assign(20, NAN);
          return kpm_moments(&km, 1, &up, &a, &b, 0.025, 20, 20, 5, 0, precision, mu.data(), nullptr, nullptr, 0,
                             nullptr, 0, nullptr);
        });
      }
  for (int precision : {KPM_FP64, KPM_FP32}) {
    const Model m(8, false);
    const kpm_spin_model sm{8, (int32_t)m.J.size(), 3, 0, m.bi.data(), m.bj.data(), m.J.data()};
    const int32_t Q = 12;
    const double a = 60.0, b = 0.0;
    check(precision == KPM_FP64 ? "spin-0" : "spin-1", [&](std::vector<double> &mu) {
      mu.assign(20, NAN);
      return kpm_spin_moments(&sm, 1, &Q, &a, &b, 20, 20, 5, 0, precision, mu.data(), nullptr, nullptr, 0, nullptr);
    });
  }
  // The gradient's fixed-point sweep needs four vectors; the checkpoints of the FP64 sweep
  // (K = 200: eight more) are not to be asked for.
  {
    const int n = 14, K = 200, R = 20;
    const Model m(n, false);
    const kpm_model km = m.of(n);
    const int32_t up = n / 2;
    std::vector<int32_t> cls(km.n_bonds);
    for (int b = 0; b < km.n_bonds; ++b) cls[b] = b / n;
    std::vector<double> g(K);
    for (int k = 0; k < K; ++k) g[k] = std::cos(1.0 + k);
    const size_t vec = (size_t)kpm_sector_dim(n, up) * R * 8;
    for (double a : {30.0, 1.0}) {  // (the second leaves the range: the FP64 sweep needs them)
      const double b = 0.0;
      check(a > 1.0 ? "gradient-inside" : "gradient-outside", [&](std::vector<double> &d) {
        d.assign(2, NAN);
        return kpm_moments_backward(&km, cls.data(), 2, 1, &up, &a, &b, K, R, 5, 0, KPM_FP64, 0, g.data(), nullptr,
                                    nullptr, d.data(), 0, nullptr, 0, nullptr);
      }, 7 * vec);
    }
  }
  return 0;
}

// Prints, for the runs given on the standard input, which form of the step libkpm
// prepares, so that tests/test_routes_host.py can check the rules of the dispatch.
// A run: n_sites R K precision n_sectors n_up... n_bonds (i j J)...
#include <cstdio>
#include <vector>

#include "kpm_run.h"

int main() {
  int N, R, K, precision, ns, nb;
  while (std::scanf("%d %d %d %d %d", &N, &R, &K, &precision, &ns) == 5) {
    std::vector<int32_t> up(ns);
    for (auto &k : up)
      if (std::scanf("%d", &k) != 1) return 1;
    if (std::scanf("%d", &nb) != 1) return 1;
    std::vector<int32_t> bi(nb), bj(nb);
    std::vector<double> J(nb);
    for (int b = 0; b < nb; ++b)
      if (std::scanf("%d %d %lf", &bi[b], &bj[b], &J[b]) != 3) return 1;
    kpm_model m{N, nb, bi.data(), bj.data(), J.data()};
    kpm::MomentsRun r;
    const int rc = kpm::prepare_run(&m, ns, up.data(), K, R, precision, &r);
    kpm::Knobs fp64;  // the same without fixed point
    fp64.fixed = 0;
    kpm::MomentsRun p;
    if (kpm::prepare_run(&m, ns, up.data(), K, R, precision, &p, fp64) != rc) return 1;
    std::printf("%d small %d fixed %d weighted %d stride %d unit %lld fp64_stride %d\n", rc, r.small,
                r.fixed, r.weighted, r.list_stride, (long long)r.fx_unit, p.list_stride);
  }
  return 0;
}

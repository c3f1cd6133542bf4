// The plan of a window of one runner m-tile, in closed form, against the
// search over every (GM, gv) that the general rule makes: prints the number of
// plans and of those that differ.
#include <cstdio>

#include "common.cuh"

using namespace bd;

static void search(const BandPlan& p, int n_rows, int* gm_out, int* gv_out) {
  const int n_mt = plan_runner_mts(p, n_rows) > 0 ? plan_runner_mts(p, n_rows) : 1;
  int glo, ghi, vlo, vhi;
  plan_gm_range(p, plan_bm(p, n_rows), n_mt, &glo, &ghi);
  plan_gv_range(p, &vlo, &vhi);
  uint64_t least = ~uint64_t(0), best = ~uint64_t(0);
  for (int gm = glo; gm <= ghi; ++gm)
    for (int gv = vlo; gv <= vhi; ++gv) least = plan_cost(p, n_mt, gm, gv) < least ? plan_cost(p, n_mt, gm, gv) : least;
  for (int gm = glo; gm <= ghi; ++gm)
    for (int gv = vlo; gv <= vhi; ++gv) {
      const uint64_t c = plan_cost(p, n_mt, gm, gv);
      if (c > least + least / MAKESPAN_SLACK_DIV) continue;
      const uint64_t k = plan_key(p, n_mt, gm, gv, c);
      best = k < best ? k : best;
    }
  *gm_out = static_cast<int>(best & 1023u);
  *gv_out = static_cast<int>((best >> 10) & 1023u);
}

int main() {
  long n = 0, differ = 0;
  for (int G = 1; G <= 460; G += G < 40 ? 1 : 7)
    for (int n_vt = 1; n_vt < 1300; n_vt += n_vt < 100 ? 1 : 13)
      for (int fixed : {0, 1, 5, 400})
        for (int bm : {int(BM_PAIR), int(BM_QUANT), 128}) {
          BandPlan p{};
          p.BM = bm;
          p.G = G;
          p.n_vt = n_vt;
          p.cpu = 2;
          p.mc = 1;
          p.row_bytes = 4096;
          p.gv_fixed = fixed;
          int gm, gv, gm1 = 0, gv1 = 0;
          search(p, 100, &gm, &gv);
          ++n;
          if (!plan_single(p, 1, &gm1, &gv1) || gm != gm1 || gv != gv1) ++differ;
        }
  BandPlan two{};
  int gm, gv;
  if (plan_single(two, 2, &gm, &gv)) ++differ;  // more m-tiles: the general rule
  std::printf("%ld %ld\n", n, differ);
  return 0;
}

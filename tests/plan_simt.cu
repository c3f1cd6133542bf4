// The row groups of the SIMT kernel over the sizes that the entry points take: prints the number of plans and of those
// whose groups do not cover the rows or are none the kernel has. Built with signed overflow trapping.
#include <cstdio>

#include "common.cuh"

using namespace bd;

int main() {
  long n = 0, bad = 0;
  for (int n_rows = 1; n_rows <= 1 << 24; n_rows += n_rows < 7000 ? 13 : n_rows / 3)
    for (int n_vt : {1, 3, 76, 450, 1573, 100000, 9586981})
      for (int G : {304, 456}) {
        BandPlan p{};
        p.BM = BM_SIMT;
        p.G = n_vt < 100 ? 2 * n_vt : G;
        p.n_vt = n_vt;
        const int rows = simt_group_rows(p, n_rows);
        ++n;
        if (rows < 1 || rows > 96 || rows % (rows <= 64 ? 8 : 16) != 0 || cdiv(n_rows, rows) > cdiv(n_rows, 96) + 3) ++bad;
      }
  std::printf("%ld %ld\n", n, bad);
  return 0;
}

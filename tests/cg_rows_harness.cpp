// Host-only: rings of n rows with ``k`` neighbours each, partitioned for the
// FP32 CG, and the number of entries its kernels gather at once. Prints
// "k degree lw row_max wide".
#include <cstdio>
#include <vector>

#include "emu_cgpart.h"

int main() {
  const int64_t n = 600;
  for (int k : {2, 6, 8, 14})
    for (int degree : {1, 4}) {
      std::vector<double> Q(3 * n, 0.0), val;
      std::vector<int32_t> rowptr(1, 0), col;
      for (int64_t v = 0; v < n; ++v) {
        Q[3 * v] = (double)v;
        for (int d = -k / 2; d <= k / 2; ++d) {
          col.push_back((int32_t)((v + d + n) % n));
          val.push_back(d == 0 ? k + 1.0 : -1.0);
        }
        rowptr.push_back((int32_t)col.size());
      }
      emu::CgPartHost P;
      if (!emu::build_cg_partition(n, Q.data(), rowptr, col, val, 2, 2, 256, degree, &P)) return 1;
      printf("%d %d %d %d %d\n", k, degree, P.lw, P.row_max, emu::cg_wide_rows(P.lw, P.row_max) ? 1 : 0);
    }
  return 0;
}

// Lists of long rows for more patterns than one page of counts holds: list q
// is of a matrix of 200 rows whose row q alone is long.  Prints "ok" when every
// list names its row and when a page's last and first lists are right.
#include <cstdio>
#include <vector>

#include "kernels.h"

int main() {
  using namespace scr;
  constexpr int kRows = 200, kLists = 130, kLong = 40;  // more than max(32, 3 x the mean)
  try {
    DeviceArena a(0);
    LongRows lr(a, 0);
    for (int q = 0; q < kLists; ++q) {
      std::vector<int> rp(kRows + 1, 0);
      for (int i = 0; i < kRows; ++i) rp[i + 1] = rp[i] + (i == q ? kLong : 1);
      int* d = a.alloc<int>(kRows + 1);
      SCR_CUDA(cudaMemcpy(d, rp.data(), sizeof(int) * (kRows + 1), cudaMemcpyHostToDevice));
      if (lr.add(kRows, rp[kRows], d) != q) return 1;
    }
    lr.read();
    for (int q = 0; q < kLists; ++q) {
      DBsr<double> M;
      lr.set(q, M);
      int row = -1;
      if (M.nlong == 1) SCR_CUDA(cudaMemcpy(&row, M.lrow, sizeof row, cudaMemcpyDeviceToHost));
      if (M.nlong != 1 || M.lthr != 32 || row != q) {
        printf("list %d: %d rows, first %d, threshold %d\n", q, M.nlong, row, M.lthr);
        return 1;
      }
    }
  } catch (const CudaError& e) {
    printf("error: %s\n", e.where);
    return 1;
  }
  printf("ok\n");
  return 0;
}

// Host driver: the tets of each warp of the element pass.  Reads "nt block_threads",
// prints how many tets the warps of all blocks cover and the end of the last record
// written.
#include <cstdio>

#include "../../paper_1506_07577_gb300/csrc/row_matrix.cuh"

int main() {
  int nt, threads;
  while (scanf("%d %d", &nt, &threads) == 2) {
    long sum = 0, end = 0;
    for (int b = 0; b < (nt + threads - 1) / threads; ++b)
      for (int w0 = 0; w0 < threads; w0 += 32) {
        const int t0 = b * threads + w0, n = ebb::warp_tets(t0, nt);
        sum += n;
        if (n > 0 && t0 + n > end) end = t0 + n;
      }
    printf("%ld %ld\n", sum, end);
  }
  return 0;
}

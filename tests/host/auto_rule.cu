// Host driver: EBB_REDUCE_AUTO of untuned FP64 maps.  Reads pairs "tets most_tets".
#include <cstdio>

#include "../../paper_1506_07577_gb300/csrc/ebb_internal.h"

int main() {
  long long tets;
  int most;
  while (scanf("%lld %d", &tets, &most) == 2) printf("%d\n", (int)ebb::auto_reduce_f64(tets, most));
  return 0;
}

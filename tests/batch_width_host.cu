// Host program around the batch-width rule of host-driven batches: lines "acc trials u tail K" give the
// width.
#include <cstdio>

#include "mca_internal.h"

int main() {
  float acc, trials, u, tail;
  int K;
  while (std::scanf("%f %f %f %f %d", &acc, &trials, &u, &tail, &K) == 5)
    std::printf("%d\n", mca::batch_width_waves(acc, trials, u, tail, K));
  return 0;
}

// Trial-loop and evaluation variants for identity outputs with softmax cross-entropy.
#include "mca_mlp2.cuh"

namespace mca {

LoopFn loop_variant_ce(LoopKind kind, int act1, int C) {
  if (C == 10) return loop_variant<MCA_ACT_IDENTITY, MCA_LOSS_SOFTMAX_CE, 10, 10>(kind, act1);
  if (C < 10) return loop_variant<MCA_ACT_IDENTITY, MCA_LOSS_SOFTMAX_CE, -1, 10>(kind, act1);
  return loop_variant<MCA_ACT_IDENTITY, MCA_LOSS_SOFTMAX_CE, -1, 14>(kind, act1);
}

}  // namespace mca

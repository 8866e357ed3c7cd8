// Trial-loop and evaluation variants for sigmoid outputs with the MSE loss.
#include "mca_mlp2.cuh"

namespace mca {

LoopFn loop_variant_mse(LoopKind kind, int act1, int C) {
  if (C == 10) return loop_variant<MCA_ACT_SIGMOID, MCA_LOSS_MSE_ONEHOT, 10, 10>(kind, act1);
  if (C < 10) return loop_variant<MCA_ACT_SIGMOID, MCA_LOSS_MSE_ONEHOT, -1, 10>(kind, act1);
  return loop_variant<MCA_ACT_SIGMOID, MCA_LOSS_MSE_ONEHOT, -1, 14>(kind, act1);
}

}  // namespace mca

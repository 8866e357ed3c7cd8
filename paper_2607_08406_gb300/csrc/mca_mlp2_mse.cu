// Trial-loop variants for sigmoid outputs with the MSE loss.
#include "mca_mlp2.cuh"

namespace mca {

LoopFn loop_variant_mse(bool window, int act1, bool ten) {
  return ten ? loop_variant<MCA_ACT_SIGMOID, MCA_LOSS_MSE_ONEHOT, 10>(window, act1)
             : loop_variant<MCA_ACT_SIGMOID, MCA_LOSS_MSE_ONEHOT, -1>(window, act1);
}

}  // namespace mca

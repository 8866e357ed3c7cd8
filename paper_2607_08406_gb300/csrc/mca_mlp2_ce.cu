// Trial-loop variants for identity outputs with softmax cross-entropy.
#include "mca_mlp2.cuh"

namespace mca {

LoopFn loop_variant_ce(bool window, int act1, bool ten) {
  return ten ? loop_variant<MCA_ACT_IDENTITY, MCA_LOSS_SOFTMAX_CE, 10>(window, act1)
             : loop_variant<MCA_ACT_IDENTITY, MCA_LOSS_SOFTMAX_CE, -1>(window, act1);
}

}  // namespace mca

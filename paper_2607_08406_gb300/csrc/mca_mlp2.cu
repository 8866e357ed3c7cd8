// Variants of the single-hidden-layer trial loop (mca_mlp2.cuh), their choice and their launch.
#include "mca_mlp2.cuh"

namespace mca {

size_t mlp2_window_smem_bytes(int RS) { return window_smem_bytes(RS); }

// Kernel variants. The output transfer function with the loss (sigmoid and MSE; identity and
// softmax cross-entropy), the hidden transfer function (tanh, Gaussian, ReLU) and 10 classes are
// fixed at compile time; everything else takes run-time switches, which cost most in the windowed
// loop, whose batch is one long instruction sequence: with them a batch took 14.6 us for a 7-class
// Gaussian net of 1001 hidden neurons and 17.0 us for 2048 ReLU neurons under the Metropolis rule;
// the variants (with the producers computing the rule's threshold) took 4.5 and 4.2 us, and take 3.3 and
// 3.7 with what came since. The variants of each loss are compiled in their own file.
static LoopKind loop_kind(const Mlp2Args& a) {
  if (a.n_explicit > 0) return a.smem_records ? kLoopEval : kLoopTrial;
  return a.window ? kLoopWindow : kLoopTrial;
}

static LoopFn pick_loop(const Mlp2Args& a) {
  const LoopKind kind = loop_kind(a);
  if (a.act2 == MCA_ACT_SIGMOID && a.loss == MCA_LOSS_MSE_ONEHOT)
    return loop_variant_mse(kind, a.act1, a.C);
  if (a.act2 == MCA_ACT_IDENTITY && a.loss == MCA_LOSS_SOFTMAX_CE)
    return loop_variant_ce(kind, a.act1, a.C);
  return loop_kernel<-1, -1, -1, -1, 14>(kind);
}

size_t mlp2_loop_smem_bytes(const Mlp2Args& a) {
  if (a.window && a.n_explicit == 0) return mlp2_window_smem_bytes(a.RS);
  return a.smem_records ? (size_t)a.RS * kRecFields * sizeof(float) : 0;
}

int mlp2_loop_max_grid(const Mlp2Args& a, int num_sms) {
  const LoopFn loop = pick_loop(a);
  const size_t smem = mlp2_loop_smem_bytes(a);
  if (smem > 0 && cudaFuncSetAttribute((const void*)loop,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem) != cudaSuccess)
    return 0;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, loop, kLoopThreads, smem) !=
      cudaSuccess)
    return 0;
  return occ * num_sms;
}

cudaError_t launch_mlp2_loop(const Mlp2Args& a, cudaStream_t s) {
  const LoopFn loop = pick_loop(a);
  const size_t smem = mlp2_loop_smem_bytes(a);
  if (smem > 0) {
    cudaError_t e = cudaFuncSetAttribute((const void*)loop,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  Mlp2Args args = a;
  void* params[] = {&args};
  if (loop_kind(a) == kLoopEval)     // no CTA waits for another
    return cudaLaunchKernel((const void*)loop, dim3(a.NR), dim3(kEvalThreads), params, smem, s);
  return cudaLaunchCooperativeKernel((const void*)loop, dim3(a.NR), dim3(kLoopThreads), params,
                                     smem, s);
}

}  // namespace mca

// Internal declarations shared by the C-ABI layer (mca_api.cu) and the kernels.
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/mca.h"

namespace mca {

struct GridBarrier;

constexpr int kKmax = 128;        // speculative candidates per batch
constexpr int kMaxC = 14;         // output fields a sample record holds
constexpr int kSR = 16;           // fields per sample record: outputs [0, C), loss 14, label 15
constexpr int kMaxClasses = kSR - 2;
constexpr int kLoopThreads = 512; // threads per CTA of the trial-loop kernel
constexpr int kLoopWarps = kLoopThreads / 32;
constexpr int kMaxSubs = 8;       // sub-chunks of one candidate inside one sample range
constexpr int kRangeTarget = 64;
// Batch width of the single-hidden-layer loop: ceil(c / p) candidates, p = (A + 0.5) / (T + 1) from
// counts decayed per batch.
constexpr float kRateDecay = 0.95f;
// In the windowed loop kWidthMlp2Long where a feature has more than one chunk of 32 entries per range: a batch
// of seven live candidates has one warp each, which takes a round of chunks more than six with two
// warps. 784-16384-10 on 60000 samples, trials 375k .. 1M (p = 0.29): 691k trials/s at 2, 714k at 1.6,
// 716k at 1.4; trials 0 .. 4000 (p = 0.48): 8.11, 7.92 and 8.11 ms.
constexpr float kWidthMlp2 = 2.0f, kWidthMlp2Long = 1.6f;
// Host-driven batches (deep nets, the Transformer): a batch of K candidates consumes
// (1 - (1 - p)^K) / p trials on average and costs about r + K candidate evaluations, r being its
// fixed part (decision, adoption or commit, launch gaps, the last partial wave of CTAs). The width
// maximises trials per cost.
inline int batch_width_cost(float acc, float trials, float r, int K) {
  const double p = ((double)acc + 0.5) / ((double)trials + 1.0);
  double qk = 1.0, best = -1.0;
  int kb = 1;
  for (int k = 1; k <= K; ++k) {
    qk *= 1.0 - p;
    const double v = (1.0 - qk) / ((double)r + (double)k);
    if (v > best) {
      best = v;
      kb = k;
    }
  }
  return kb;
}

// The same with the grid's size: a candidate's CTAs fill the fraction u of the GPU, so that candidates
// cost nothing more until the GPU is full, and then u each (a: what the last, partial wave costs).
// In units of one CTA's chain: r + max(1, a + K u). Measured on GB300 with fixed widths: for 24 x 256
// tanh nets on 10000 samples (u = 0.52) 177, 283, 362, 431, 575 us per batch at K = 1, 2, 3, 4, 6, that
// is 135 (0.3 + max(1, 0.7 + K u)) within 5 %; for the d_model 128 Transformer on 256 sequences (u = 0.84) 116,
// 200, 274, 350, 491, that is 89 (0.3 + max(1, 0.15 + K u)). Small nets (u < 1/4) gain most: at an
// acceptance of one half they consume 1.9 trials per batch instead of 1 to 1.5.
constexpr float kWaveFixed = 0.3f;
constexpr float kWaveTailDeep = 0.7f;
constexpr float kWaveTailTfm = 0.15f;

inline int batch_width_waves(float acc, float trials, float u, float tail, int K) {
  if (u > 1.0f) return batch_width_cost(acc, trials, (kWaveFixed + tail) / u, K);
  const double p = ((double)acc + 0.5) / ((double)trials + 1.0);
  double qk = 1.0, best = -1.0;
  int kb = 1;
  for (int k = 1; k <= K; ++k) {
    qk *= 1.0 - p;
    const double fill = (double)k * (double)u;
    const double t = (double)kWaveFixed + (fill <= 1.0 ? 1.0 : (double)tail + fill);
    const double v = (1.0 - qk) / t;
    if (v > best) {
      best = v;
      kb = k;
    }
  }
  return kb;
}
constexpr int kSmemRecordBytes = 160 * 1024;  // larger ranges keep their records in global memory
// Window of the trial loop: kWS candidate slots per CTA, each caching up to kCap entries of the
// candidate's segment (range-local sample, activation change, new hidden field), prepared ahead of
// the batches. Batches are at most kWinBatch wide.
constexpr int kWS = 96;
constexpr int kCap = 160;
constexpr int kWinBatch = 64;
// Per-batch accumulator buffer of the windowed loop: one packed word per candidate (arrival count
// in bits 56..63, count of out-of-range shares in 48..55, fixed-point sum below), kAccWord words
// apart, so that the CTAs' additions to a batch's candidates go to different lines (and L2 slices)
// instead of queueing at one. Four buffers rotate. One warp reads a batch's words, two per lane; the
// count fields cap the ranges at 255.
constexpr int kAccWord = 32;
constexpr int kArrivalWord = 64;   // count-only word of a batch without a live candidate
constexpr int kAccStride = (kArrivalWord + 1) * kAccWord;
constexpr int kAccBuffers = 4;
constexpr int kWindowMaxRanges = 255;
static_assert(kWinBatch <= 64 && kWinBatch < kWS, "a windowed batch is read by one warp, two per lane");

// Device-resident run state (one per handle).
struct DevState {
  double S;                  // loss sum of the cached state
  unsigned long long trials, accepts, candidates, batches, wasted, forced, trace_written;
  unsigned long long alg_bytes;  // compulsory DRAM bytes of the evaluated candidates and commits
  unsigned long long phase_ns[8];  // CTA 0: set-up, evaluate, arrive, wait, reduce+decide, commit;
                                   // [6] wait averaged over all CTAs
  unsigned long long alg_flops;    // deep path: FLOPs of the evaluated candidates' chains
  float rate_acc, rate_trials;     // decayed counts of accepts and trials (batch-width choice)
  int err;                   // first device-side error (mca_status), 0 = none
  int pad;
};

// The candidates of an explicit evaluation, copied to the device in one piece.
struct ExCands {
  unsigned int idx[kKmax];
  float new_w[kKmax];
};

// What an explicit evaluation reports beside its loss changes.
struct ExTail {
  double S;                  // loss sum of the cached state
  int err;                   // first device-side error
};

// Arguments of the two-layer trial loop (input -> hidden -> output). The samples are split into NR
// contiguous ranges of RS samples (RS a multiple of 8); CTA r owns range r.
struct Mlp2Args {
  int N, D, H, C, Np;
  int NR, RS, SUB;           // ranges, samples per range, entries per sub-chunk (multiple of 32)
  int smem_records;          // 1: each CTA keeps its range's sample records in shared memory
  int window;                // 1: run the windowed trial loop (records and window in shared memory)
  float wscale;              // the windowed loop's batches take ceil(wscale / p) candidates
  unsigned long long P, P1;
  const int* xs_off;         // [D + 1] CSR of X by feature: entries of feature i in [off[i], off[i+1])
  const int* xs_n;           // [nnz] sample index of each entry (ascending inside a feature)
  const float* xs_v;         // [nnz] value x[n, i] != 0
  const int* xs_sect;        // [D] 32-byte sectors of a z1 row that feature i's entries touch
  const int* xs_roff;        // [D x (NR + 1)] first entry of feature i in range r
  float* z1;                 // [H x Np] hidden fields, feature-major
  float* srec;               // [kSR x Np] field-major: output fields, loss, label
  float* w1;                 // [H x D] effective weights
  float* w2;                 // [C x H]
  signed char* code1;        // ternary codes / mask bits (nullable for fp32 layers)
  signed char* code2;
  const float* wfix1;        // masked layers: fixed weights
  const float* wfix2;
  int wk1, wk2;
  float sc1, sc2;
  int act1, act2;
  float g1, g2;
  int loss;
  int op;
  float lo, hi, delta, bound;
  int strict;
  int metro;                 // 1: Metropolis rule (Eq. 7) with msc = N / beta; 0: greedy (Eq. 6)
  double msc;
  int stretch;               // > 0: current-layer schedule, trials per stretch; 0: uniform index
  unsigned long long seed, tau0, n_trials;
  int K;
  int fixed_K;
  float* partial;            // [2 x kKmax x NR] per-candidate, per-range loss changes
  unsigned long long* accum; // [kAccBuffers x kAccStride] windowed loop: fixed-point sums, counts, arrivals
  GridBarrier* bar;
  DevState* st;
  mca_trace_rec* trace;
  int trace_cap;
  const unsigned long long* ftau;
  const unsigned char* facc;
  int nforce;
  int n_explicit;            // > 0: evaluate these candidates once, no decision, no commit
  const unsigned int* ex_idx;
  const float* ex_new;
  double* ex_out;
  ExTail* ex_tail;           // nullable
};

// ------------------------------------------------------------------------------------------------
// Deep MLP path (three or more weight layers): every layer's fields are cached; a candidate in layer
// l updates row j of layer l, then layer l+1 by one weight column (rank-1), then recomputes the layers
// from l+2 on as  Z'_m = Z_m + W_m (f(Z'_{m-1}) - f(Z_{m-1}))  over tiles of kDeepTS samples.
// ------------------------------------------------------------------------------------------------
constexpr int kMaxLayers = 32;
constexpr int kDeepTS = 64;        // samples per tile of the SIMT chain, or
constexpr int kDeepSmallTS = 32;   //   of small nets (deep_tile_samples)
constexpr int kTcTS = 128;         // samples per tile of the tensor-core chain (one MMA M)
constexpr int kDeepThreads = 256;
constexpr int kDeepMaxWidth = 256; // widths of the layers inside the dense chain
constexpr int kDeepKC = 16;        // weight-tile depth of the chain GEMM
constexpr float kDeepDScale = 16384.0f;   // tanh changes (at most 2) as fp16 operands: scale
// Two fp16 parts of a value hold its 22 leading bits, like two tf32 parts, down to 2^-17 of the power of two
// that its operand is scaled for; below, their error is absolute, 2^-40 of that power. So an operand is
// taken as fp16 parts only while at most wide_allowance of a row's n non-zero entries lie below 2^-17:
// of uniform values 2^-17 do, 0.03 in a row of 256 weights of +-0.1 under a bound of 2.
constexpr int kWideGap = 17;
constexpr unsigned int wide_allowance(unsigned int n) { return 3u + n / 2048u; }
constexpr int kDeepScrSlots = 16;  // candidates whose fields the tensor-core evaluation keeps
constexpr float kTfmF16Max = 4.0f;   // largest parameter magnitude of the fp16 Transformer kernels
constexpr float kTfmF16Min = 0x1p-10f;   // ... and the smallest that their scales follow
constexpr int kTfmScrSlots = 16;   // candidates whose residual streams the evaluation keeps
constexpr size_t kSimtScrBytes = (size_t)1 << 30;   // all slots of a SIMT evaluation

struct DeepCand {
  unsigned int idx;
  int layer, row, col;
  float oldw, neww, delta;
  int new_code, valid;
};

// Decision of the last batch, written by the decide kernel and read by the commit kernel and host.
struct DeepCtl {
  int kstar;                 // accepted candidate, -1 none, -2 non-finite loss change
  int consumed;              // trials consumed by the batch
  DeepCand acc;              // the accepted candidate
};

struct DeepArgs {
  int L, N, Np, D, C, ntiles;
  int n_in[kMaxLayers], n_out[kMaxLayers], act[kMaxLayers], wk[kMaxLayers];
  float g[kMaxLayers], sc[kMaxLayers];
  unsigned long long off[kMaxLayers + 1];
  float* w[kMaxLayers];
  signed char* code[kMaxLayers];
  const float* wfix[kMaxLayers];
  float* Z[kMaxLayers];      // [n_out[l] x Np] fields of layer l; Z[L-1] are the output fields
  float* whi[kMaxLayers];    // tensor-core chain: tf32(W_m) and tf32(W_m - tf32(W_m)) of the
                             //   256 x 256 layers 1 .. L-2 as stage images (null otherwise)
  int tile;                  // samples per tile
  int tc;                    // 1: dense chain on the tensor cores, tiles of kTcTS samples
  int tc_f16;                // tc = 1: operands as fp16 parts (tanh layers), else tf32 parts
  float tc_wscale;           // tc_f16: power of two that scales the dense weights to at most 2^15
  float tc_dscale;           // tc_f16: 1 / (tc_wscale kDeepDScale), the products' scale
  const float* XT;           // [D x Np]
  float* ell;                // [Np] per-sample loss
  const int* y;
  int loss;
  int op;
  float lo, hi, delta, bound;
  int strict;
  int metro;                 // 1: Metropolis rule (Eq. 7) with msc = N / beta; 0: greedy (Eq. 6)
  double msc;
  int stretch;               // > 0: current-layer schedule, trials per stretch; 0: uniform index
  unsigned long long seed, tau;
  int Kb;
  float* partial;            // [kKmax x ntiles]
  DevState* st;
  DeepCtl* ctl;
  mca_trace_rec* trace;
  int trace_cap;
  const unsigned long long* ftau;
  const unsigned char* facc;
  int nforce;
  int n_explicit;
  const unsigned int* ex_idx;
  const float* ex_new;
  double* ex_out;
  ExTail* ex_tail;           // nullable
  // evaluation of candidate k < nscr (on the tensor cores with a dense chain, layer <= L-3): every field it
  // computes goes to scr[k * (L + 1) + m] (layer m: row j of the mutated layer, the full layers
  // after it; m = L: the per-sample losses), so that an accepted candidate's fields are adopted instead
  // of recomputed (tensor-core chain: by swapping pointers, SIMT chain: by a copy)
  float* const* scr;
  int nscr;
};

cudaError_t launch_deep_eval(const DeepArgs& a, cudaStream_t s);    // grid (Kb, ntiles)
int deep_eval_ctas_per_sm(const DeepArgs& a);
cudaError_t launch_deep_decide(const DeepArgs& a, cudaStream_t s);  // one CTA
cudaError_t launch_deep_commit(const DeepArgs& a, cudaStream_t s);  // grid ntiles
cudaError_t launch_deep_forward_layer(const DeepArgs& a, int l, cudaStream_t s);
cudaError_t launch_deep_losses(const DeepArgs& a, cudaStream_t s);
cudaError_t launch_deep_split(const DeepArgs& a, cudaStream_t s);     // W_hi / W_lo of all layers
// *top = bits of the dense weights' largest magnitude (of those behind the masks), at least its old value.
cudaError_t launch_deep_top(const DeepArgs& a, int* top, cudaStream_t s);
// *out = 1 if the dense weights are out of the fp16 parts' range under the bound pow2_above(max(*top,
// floor)); top: bits of a float >= 0, or null. (*out is left alone otherwise.)
cudaError_t launch_deep_wide(const DeepArgs& a, const int* top, float floor, int* out,
                             cudaStream_t s);
cudaError_t launch_deep_eval_tc(const DeepArgs& a, cudaStream_t s);   // grid (Kb, ntiles)
cudaError_t launch_deep_commit_tc(const DeepArgs& a, cudaStream_t s); // grid ntiles
cudaError_t launch_deep_forward_tc(const DeepArgs& a, cudaStream_t s);  // grid ntiles

// ------------------------------------------------------------------------------------------------
// Character-level Transformer path: pre-LN GPT blocks over B sequences of T tokens. All parameters
// live in one flat fp32 array; a candidate recomputes each sequence from the first stage its
// parameter feeds (embeddings, block b, or the final LN and head), reading the parameters through
// a one-element patch (index midx reads mval), on the cached residual stream at that stage.
// ------------------------------------------------------------------------------------------------
constexpr int kTfmMaxBlocks = 8;
constexpr int kTfmThreads = 512;
constexpr int kTfmMaxT = 64;
constexpr int kTfmMaxD = 128;
constexpr int kTfmMaxV = 128;
constexpr int kTfmFC = 128;        // FFN hidden columns per chunk

enum TfmMode { kTfmEval = 0, kTfmCommit = 1, kTfmForward = 2 };

struct TfmArgs {
  int V, T, d, H, dh, F, nL, B;
  float eps;
  int act;
  float g;
  // flat offsets: embeddings, the first block, the block stride, the final LN and the head; and the
  // offsets inside a block
  unsigned long long o_tok, o_pos, o_blk0, blk_size, o_lnf_g, o_lnf_b, o_wh, o_bh, P;
  unsigned int r_ln1g, r_ln1b, r_wq, r_bq, r_wk, r_bk, r_wv, r_bv, r_wo, r_bo, r_ln2g, r_ln2b,
      r_w1, r_b1, r_w2, r_b2;
  float* params;             // [P]
  const int* tokens;         // [B x (T + 1)]
  float* X;                  // [(nL + 1) x B x T x d] residual stream entering block b (b = nL: final)
  float* Xmid;               // [nL x B x T x d] block b's stream after its attention sub-block (tc)
  float* ell;                // [B] per-sequence loss sums
  int loss_unused;
  int op;
  float lo, hi, delta, bound;
  int strict;
  int metro;                 // 1: Metropolis rule (Eq. 7) with msc = N / beta; 0: greedy (Eq. 6)
  double msc;
  int stretch;               // > 0: current-layer schedule, trials per stretch; 0: uniform index
  unsigned long long seed, tau;
  int Kb;
  int mode;
  size_t smem;               // dynamic shared memory of the sequence kernel
  float* partial;            // [kKmax x B]
  DevState* st;
  DeepCtl* ctl;
  mca_trace_rec* trace;
  int trace_cap;
  const unsigned long long* ftau;
  const unsigned char* facc;
  int nforce;
  int n_explicit;
  const unsigned int* ex_idx;
  const float* ex_new;
  double* ex_out;
  ExTail* ex_tail;           // nullable
  int tc;                    // 1: the tensor-core kernels (mca_tfm_tc.cu) run the sequences
  float* wimg;               // their split-weight images (mca_tc_layout.h), tc = 1 only
  void* wimg16;              // the images with fp16 parts, kept beside them
  int f16;                   // tc = 1: run the kernels with fp16 parts (every parameter, and every
                             //   candidate's, at most kTfmF16Max in magnitude), with
  float f16_w, f16_ln, f16_act;   //   these scales (powers of two) of the weights in wimg16, of layer-norm
  float f16_dln, f16_dact;        //   outputs and of other activations; the products' scales back
  // scratch slots (trial loop only): candidate k < nscr of a batch writes the residual streams it
  // recomputes to slot k of scrX ([nscr][(2 nL + 1) x B x T x d]: X, then Xmid; SIMT: X alone) and its
  // sequence losses to scr_ell ([nscr][B]); an accepted candidate with a slot is adopted from it
  float* scrX;
  float* scr_ell;
  int nscr;
  // batches run ahead of the host (tc = 1, trial loop): the batch's first trial is read from
  // tau_dev, which the decision advances by the trials it consumed; trials at or past tau_end do not
  // exist (a batch that starts there does nothing). nullptr: the batch starts at tau.
  unsigned long long* tau_dev;
  unsigned long long tau_end;
};

size_t tfm_smem_bytes(int T, int d, int dh, int V);
int tfm_eval_ctas_per_sm(const TfmArgs& a);
cudaError_t launch_tfm_eval(const TfmArgs& a, cudaStream_t s);      // grid (Kb, B)
cudaError_t launch_tfm_decide(const TfmArgs& a, cudaStream_t s);    // one CTA
cudaError_t launch_tfm_commit(const TfmArgs& a, cudaStream_t s);    // grid B
cudaError_t launch_tfm_forward(const TfmArgs& a, cudaStream_t s);   // grid B, writes every stage
// Tensor-core Transformer kernels (two sequences per CTA): the split-weight images from the
// parameters, the three sequence modes, and the image entry of the accepted parameter after a commit.
cudaError_t launch_tfm_tc_split(const TfmArgs& a, cudaStream_t s);
cudaError_t launch_tfm_f16_split(const TfmArgs& a, cudaStream_t s);
// *out = 1 if parameters are too small for the fp16 parts at level q (bound: of the activations there).
cudaError_t launch_tfm_f16_range(const TfmArgs& a, float q, float bound, int* out, cudaStream_t s);
cudaError_t launch_tfm_f16(const TfmArgs& a, int mode, cudaStream_t s);   // the three modes, fp16 parts
cudaError_t launch_tfm_tc_eval(const TfmArgs& a, cudaStream_t s);      // grid (Kb, B / 2)
cudaError_t launch_tfm_tc_commit(const TfmArgs& a, cudaStream_t s);    // grid B / 2
cudaError_t launch_tfm_tc_forward(const TfmArgs& a, cudaStream_t s);   // grid B / 2
// After the commit kernel: the accepted weight's image entry and, with a scratch slot, adoption.
cudaError_t launch_tfm_tc_adopt(const TfmArgs& a, cudaStream_t s);     // grid (B, 2 nL + 1)

// Launchers (mca_mlp2.cu). All enqueue on `stream` and return the CUDA error of the launch.
cudaError_t launch_transpose_pad(const float* X, int N, int D, float* XT, int Np, cudaStream_t s);
cudaError_t launch_csr_count(const float* XT, int Np, int N, int D, int* cnt, cudaStream_t s);
cudaError_t launch_csr_fill(const float* XT, int Np, int N, int D, const int* off, int* xs_n,
                            float* xs_v, cudaStream_t s);
cudaError_t launch_csr_sectors(const int* off, const int* xs_n, int D, int* sect, cudaStream_t s);
cudaError_t launch_csr_range_offsets(const int* off, const int* xs_n, int D, int NR, int RS,
                                     int* roff, cudaStream_t s);
cudaError_t launch_count_nonfinite(const float* p, size_t n, int* out, cudaStream_t s);
// *out = max(*out, bits of max |p[i]|) (finite values; *out holds the bits of a float >= 0).
cudaError_t launch_abs_max(const float* p, size_t n, int* out, cudaStream_t s);
cudaError_t launch_init_layer(int wkind, float scale, const float* src, const signed char* mask,
                              size_t n, float* w_eff, signed char* code, float* wfix,
                              cudaStream_t s);
cudaError_t launch_sgemm_nn(int M, int Ncol, int K, const float* A, int lda, const float* B,
                            int ldb, float* C, int ldc, cudaStream_t s);
cudaError_t launch_mlp2_outputs(const Mlp2Args& a, const int* y, cudaStream_t s);
// S = sum of ell[0 .. N) in fp64 (fixed order) into st->S.
cudaError_t launch_sum_loss(const float* ell, int N, DevState* st, cudaStream_t s);
// Cooperative persistent trial loop, one CTA per sample range (grid = NR).
cudaError_t launch_mlp2_loop(const Mlp2Args& a, cudaStream_t s);
size_t mlp2_window_smem_bytes(int RS);
int mlp2_loop_max_grid(const Mlp2Args& a, int num_sms);
size_t mlp2_loop_smem_bytes(const Mlp2Args& a);

// Proposals of trials tau0 .. tau0 + n - 1 as explicit candidates (mca_propose.cu): the trial's
// record (index, effective weights before and after, validity) and the candidate arrays of the
// explicit evaluation (a rejected proposal is evaluated as the no-op).
struct ProposeArgs {
  int L, n;
  unsigned long long off[kMaxLayers + 1];   // flat offset of each layer; off[L] = P
  int wk[kMaxLayers];
  float sc[kMaxLayers];
  const float* w[kMaxLayers];
  const signed char* code[kMaxLayers];
  const float* wfix[kMaxLayers];
  int op;
  float lo, hi, delta, bound;
  int stretch;
  unsigned long long seed, tau0;
  mca_trace_rec* rec;        // [n]
  unsigned int* ex_idx;      // [n]
  float* ex_new;             // [n]
};
cudaError_t launch_propose(const ProposeArgs& a, cudaStream_t s);

// Fields of a layer on the tensor cores (mca_gemm_tc.cu): Z[M x Np] = W[M x K] act(B)[K x Np]
// (act < 0: B as it is), three MMAs per product of fp16 or tf32 parts. img: scratch of
// gemm_tc_image_bytes(M, K, Np) bytes, 256-byte aligned; err: device status word (MCA_ERR_TIMEOUT when a
// bounded wait ran out).
bool gemm_tc_ok(int M, int K, int Np);
size_t gemm_tc_image_bytes(int M, int K, int Np);
cudaError_t launch_gemm_tc(const float* W, int M, int K, const float* B, int act, float g,
                           float* Z, int Np, float* img, int* err, cudaStream_t s);

}  // namespace mca

struct mca_handle;

namespace mca {
// Kernel arguments of a handle's trial loop (its state and workspace scratch).
Mlp2Args handle_mlp2_args(mca_handle* h);

}  // namespace mca

struct mca_handle {
  std::string err;
  std::vector<mca_layer> layers;
  int loss = 0;
  mca_domain dom{};
  mca_options opt{};
  long long N = 0;
  int D = 0, C = 0, Np = 0;
  unsigned long long P = 0;
  std::vector<unsigned long long> off;   // flat offset of each layer
  cudaStream_t stream = nullptr;
  int device = 0, num_sms = 0;
  // memory
  void* ws = nullptr;
  size_t ws_bytes = 0;
  bool ws_owned = false;
  float* XT = nullptr;                   // [D x Np]
  int* y = nullptr;
  int* xs_off = nullptr;
  int* xs_n = nullptr;
  float* xs_v = nullptr;
  int* xs_sect = nullptr;
  int* xs_roff = nullptr;
  long long nnz = 0;
  int max_nnz = 0;
  std::vector<float*> w_eff;
  std::vector<signed char*> code;
  std::vector<float*> wfix;
  float* z1 = nullptr;
  float* srec = nullptr;
  // deep path
  bool deep = false;
  bool tc = false;                   // deep: dense chain on the tensor cores; Transformer: the
                                     // tensor-core sequence kernels
  // deep: the chain's operands may be fp16 parts (tanh layers); the bound of the dense weights' magnitude,
  // and whether the weights are in the range of fp16 parts under it; both as the weight images
  // were split, which is what the kernels are told
  bool tc_f16 = false;
  float wbound = 1.0f, wsplit = 1.0f;
  bool parts_f16 = false, split_f16 = false;
  std::vector<float*> Z;
  std::vector<float*> whi;           // split-weight images of layers 1 .. L-2 (tensor-core chain)
  float* ell = nullptr;
  mca::DeepCtl* ctl = nullptr;
  int ntiles = 0, tile = 0;          // deep: tiles, and their samples
  float wave = 1.0f;                 // host-driven batches: CTAs per candidate / CTAs that run at once
  float* partial = nullptr;
  unsigned long long* accum = nullptr;
  int NR = 0, RS = 0, SUB = 0, smem_records = 0, window = 0;
  mca::GridBarrier* bar = nullptr;
  mca::DevState* st = nullptr;
  mca_trace_rec* trace = nullptr;
  int trace_cap = 0;
  mca::ExCands* ex = nullptr;
  // explicit evaluations: pinned host memory that the candidates are copied from and the kernels
  // write the results to
  struct EvalHost {
    mca::ExCands in;
    double dS[mca::kKmax];
    mca_trace_rec prop[mca::kKmax];
    mca::ExTail tail;
  }* ev_host = nullptr;
  int* flag = nullptr;                   // a device word for checks that the host waits for
  float* gimg = nullptr;                 // operand images of the tensor-core forward pass
  int nscr = 0;                          // host-driven batches: candidate scratch slots
  std::vector<float*> scr;               // [nscr x (L + 1)] layer m of slot k (m = L: losses)
  float** scr_dev = nullptr;             // the same table in device memory
  cudaEvent_t ev_c[2] = {nullptr, nullptr};   // around the adoption / commit after a decision
  bool ev_c_pending = false;
  // test hook
  unsigned long long* ftau = nullptr;
  unsigned char* facc = nullptr;
  int nforce = 0;
  // host-side counters
  unsigned long long tau = 0;
  unsigned long long launches = 0, resyncs = 0;
  cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};   // per-batch kernel timing (deep, Transformer)
  // Transformer tensor-core path, batches run ahead of the host: two decision buffers (device),
  // the batch's first trial (device), their pinned host mirror, and per-buffer events
  mca::DeepCtl* ctl2 = nullptr;
  unsigned long long* tau_dev = nullptr;
  struct PipeHost {
    mca::DeepCtl ctl[2];
    unsigned long long tau;
  }* pipe_host = nullptr;
  cudaEvent_t ev_p[2][3] = {{nullptr, nullptr, nullptr}, {nullptr, nullptr, nullptr}};
  unsigned long long eval_ns = 0, rest_ns = 0;
  bool broken = false;                   // a sticky CUDA error or device timeout was seen
  float rate_acc = 0.0f, rate_trials = 0.0f;   // deep path: acceptance counts (batch width)
  // transformer path
  bool tfm = false;
  mca_tfm_spec tspec{};
  float* params = nullptr;               // [P] flat parameters
  int* tokens = nullptr;                 // [B x (ctx + 1)]
  float* X = nullptr;                    // cached residual stream at every stage
  float* tfm_img = nullptr;              // split-weight images of the tensor-core kernels (tc)
  void* tfm_img16 = nullptr;             // the same with fp16 operand parts
  float pmax = 0.0f;                     // tensor-core Transformer: largest parameter magnitude
  float tfm_q = 0.0f;                    //   level of the fp16 operands' scales, 0: tf32 kernels
  bool tfm_small = false;                //   parameters too small for them: tf32 kernels
  float* tfm_Xmid = nullptr;             // its mid streams (after each block's attention)
  float* tfm_scrX = nullptr;             // Transformer: candidate scratch slots
  float* tfm_scr_ell = nullptr;          // (h->nscr of them)
};

// Character-level Transformer on the tensor cores with fp16 operand parts: the recomputation of
// mca_tfm_tc.cu (the same rows, restarts, rank-1 terms and cached streams), with every dense
// projection as three kind::f16 MMAs per product, D = A_lo W_hi^T + A_hi W_lo^T + A_hi W_hi^T. An fp16 MMA
// covers K = 16 in the time a tf32 MMA takes for K = 8, so the projections cost half. The two parts of a
// value hold its 22 leading bits, like two tf32 parts, but fp16 has less range: the operands are
// scaled by powers of two from bounds that follow from the largest parameter magnitude q (a power of two
// at or above it), and below some size the error is absolute. With q = 1: weights down to 2^-18, 2^-40
// below; layer-norm outputs down to 2^-15, 2^-37 below; attention outputs and feed-forward activations
// (of up to 257) down to 2^-10, 2^-32 below; for q in general q, q and about q^2 times that. All of them enter the
// residual stream through a weight and a sum in fp32. The host takes these kernels only while q is at most
// kTfmF16Max; mca_tfm_tc.cu has no such bound.
//
// What bounded the tf32 kernel was not the tensor pipe but one thread deciding each MMA's operands at
// run time (155 cycles per MMA whose arithmetic takes 64), and every phase waiting for the previous
// one. Here
//   - a control warp (warp 16) issues all MMAs and weight copies from one elected thread, with the
//     shapes fixed at compile time (64 cycles per N = 128 MMA);
//   - both parts of A live in tensor memory, so shared memory holds a nine-stage weight ring;
//   - the feed-forward network runs by 64 hidden units: W1 (N = 64) two halves ahead, so that the
//     activation of half h overlaps the MMAs of W2 for half h - 1 and of W1 for half h + 1.
// The weight images are stored in the order of consumption, one 16 KB chunk per copy.
//
// Tensor memory: Q, K, V in columns 0 / 128 / 256, A (LN output or attention output, K = 128) hi in
// 384 .. 447 and lo in 448 .. 511, two fp16 per column; in the feed-forward network U of half h in
// 64 (h mod 2) .., F in 128 .., the activated half A2 hi / lo in 256 + 64 (h mod 2) .. + 31 / + 32 ..;
// the output projection and the head in 0 .. 127. During attention K and V (fp32) lie in the first
// eight stages of the ring.
//
// Waits are bounded (2 s). A wait that gives up sets a flag that makes every later wait return at
// once, so all threads run through the same barriers; the control thread drains its copies and MMAs
// (bounded) before tensor memory is released, and the CTA records MCA_ERR_TIMEOUT.
#include <cuda_fp16.h>

#include "mca_tfm_tc.cuh"

namespace mca {
namespace {

constexpr int kThreads = kTfmWorkers + 32;
constexpr int kCtlWarp = kTfmWorkers / 32;
constexpr int kStages = 9;
constexpr int kStageBytes = (int)kTfmF16Chunk;
constexpr int kXsBytes = kRows * kXLd * 4;
constexpr int kSmem = kXsBytes + kStages * kStageBytes;
constexpr uint32_t kIdN128 = tc_idesc_f16(kRows, 128), kIdN64 = tc_idesc_f16(kRows, 64);
constexpr uint32_t kColQ = 0, kColK = 128, kColV = 256, kColA = 384, kAlo = 64;
constexpr uint32_t kColU = 0, kColF = 128, kColA2 = 256, kA2lo = 32;
constexpr int kQkvChunks = 12, kAttnChunks = 16;          // chunks before Wo, before the FFN
constexpr int kHeadChunks = 4;

static_assert(kSmem + 8 * 1024 <= 227 * 1024, "shared memory of the fp16 Transformer kernel");
static_assert(2 * kRows * kD * 4 <= 8 * kStageBytes, "K and V lie in eight stages");

struct Ctx : RowCtx {
  unsigned char* ring;       // weight stages
  int b0s, nb, cpb;          // first block run, blocks run, chunks per block
  int q0, total;             // chunks of the first block that are left out, chunks run in all
  bool ffn0, unit0;          // the first block starts at its FFN; after a hidden unit's rank-1 step
};

struct Bars {
  uint64_t full[kStages], empty[kStages];
  uint64_t aready, mdone;    // A written by every row warp; a product's MMAs done
  uint64_t ufull[2], a2full[2], a2empty[2], drain;
};

// Wait for phase `parity` unless some wait of the CTA gave up before.
__device__ __forceinline__ void wait_phase(uint64_t* bar, uint32_t parity, volatile int* fail) {
  if (*fail) return;
  if (!mbar_wait(bar, parity)) *fail = 1;
}

__device__ __forceinline__ void arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// ------------------------------------------------------------------------------------ control

struct Feed {
  int nload, limit, nwait, ncommit;   // chunks requested, allowed, waited for, committed
};

// The elected thread: request chunks up to (not including) `upto`, within the limit; a stage is refilled
// once the MMAs of the chunk that held it are done.
__device__ __forceinline__ void feed(const TfmArgs& a, const Ctx& c, Bars& B, Feed& f, int upto,
                                     volatile int* fail) {
  const int end = min(upto, f.limit);
  while (f.nload < end) {
    const int x = f.nload, st = x % kStages;
    if (x >= kStages) wait_phase(&B.empty[st], (uint32_t)(x / kStages - 1) & 1u, fail);
    if (*fail) return;
    bulk_load(smem_u32(c.ring + st * kStageBytes),
              reinterpret_cast<const unsigned char*>(a.wimg16) +
                  (size_t)(c.b0s * c.cpb + c.q0 + x) * kStageBytes,
              kStageBytes, &B.full[st]);
    ++f.nload;
  }
}

// The elected thread: the MMAs of chunk f.ncommit, whose weights are N rows (128: K = 32; 64: K = 64),
// into columns d from A at columns ahi (lo part alo columns further on), then the next copies.
template <int N>
__device__ __forceinline__ void mma_chunk(const TfmArgs& a, const Ctx& c, Bars& B, Feed& f,
                                          uint32_t d, uint32_t ahi, uint32_t alo, bool first,
                                          volatile int* fail) {
  constexpr uint32_t lbo = N * 16;
  constexpr int steps = N == 128 ? 2 : 4;           // K steps of 16
  const int x = f.ncommit, st = x % kStages;
  wait_phase(&B.full[st], (uint32_t)(x / kStages) & 1u, fail);
  if (*fail) return;
  f.nwait = x + 1;
  const uint64_t w = umma_desc(smem_u32(c.ring) + (uint32_t)(st * kStageBytes), lbo, 128u);
  const uint32_t dt = c.tmem + d, ta = c.tmem + ahi;
#pragma unroll
  for (int ks = 0; ks < steps; ++ks) {
    const uint64_t whi = w + (uint64_t)(ks * 2 * (lbo / 16)), wlo = whi + kStageBytes / 32;
    const uint32_t id = N == 128 ? kIdN128 : kIdN64;
    mma_ts_f16(dt, ta + alo + 8u * ks, whi, id, first && ks == 0 ? 0u : 1u);
    mma_ts_f16(dt, ta + 8u * ks, wlo, id, 1u);
    mma_ts_f16(dt, ta + 8u * ks, whi, id, 1u);
  }
  umma_commit(&B.empty[st]);
  f.ncommit = x + 1;
  feed(a, c, B, f, x + kStages, fail);
}

// The elected thread of the control warp: every MMA of the CTA, in the order of the chunks.
__device__ __forceinline__ void control(const TfmArgs& a, const Ctx& c, Bars& B,
                                        volatile int* fail) {
  Feed f;
  f.nload = f.nwait = f.ncommit = 0;
  // loads stop at the output projection of a block whose attention step is still to come: K and V
  // take the stages
  auto wo_chunk = [&](int jb) { return jb * c.cpb - c.q0 + kQkvChunks; };
  f.limit = c.nb == 0 ? c.total
            : !c.ffn0 ? wo_chunk(0)
            : c.nb > 1 ? wo_chunk(1) : c.total;
  feed(a, c, B, f, kStages, fail);
  uint32_t pa = 0u;                  // phases of aready
  int gh = 0;                        // halves of all feed-forward networks so far
  const int nh = a.F / kHc;
  for (int jb = 0; jb < c.nb; ++jb) {
    if (!(c.ffn0 && jb == 0)) {
      wait_phase(&B.aready, pa++ & 1u, fail);
      tc_fence_after();
#pragma unroll 1
      for (int q = 0; q < kQkvChunks; ++q)
        mma_chunk<128>(a, c, B, f, kColQ + 128u * (uint32_t)(q >> 2),
                       kColA + 16u * (uint32_t)(q & 3), kAlo, (q & 3) == 0, fail);
      umma_commit(&B.mdone);
      wait_phase(&B.aready, pa++ & 1u, fail);      // the attention output (K and V are free)
      tc_fence_after();
      f.limit = jb + 1 < c.nb ? wo_chunk(jb + 1) : c.total;
      feed(a, c, B, f, f.ncommit + kStages, fail);
#pragma unroll 1
      for (int q = 0; q < 4; ++q)
        mma_chunk<128>(a, c, B, f, kColU, kColA + 16u * (uint32_t)q, kAlo, q == 0, fail);
      umma_commit(&B.mdone);
    }
    wait_phase(&B.aready, pa++ & 1u, fail);
    tc_fence_after();
    auto w1 = [&](int h) {                         // U of half h
      for (int q = 0; q < 2; ++q)
        mma_chunk<64>(a, c, B, f, kColU + 64u * (uint32_t)(h & 1), kColA + 32u * (uint32_t)q, kAlo,
                      q == 0, fail);
      umma_commit(&B.ufull[h & 1]);
    };
    w1(0);
    w1(1);
#pragma unroll 1
    for (int h = 0; h < nh; ++h, ++gh) {
      wait_phase(&B.a2full[h & 1], (uint32_t)(gh >> 1) & 1u, fail);
      tc_fence_after();
      for (int q = 0; q < 2; ++q)
        mma_chunk<128>(a, c, B, f, kColF, kColA2 + 64u * (uint32_t)(h & 1) + 16u * (uint32_t)q,
                       kA2lo, h == 0 && q == 0, fail);
      umma_commit(&B.a2empty[h & 1]);
      if (h + 2 < nh) w1(h + 2);
      if (h == nh - 1) umma_commit(&B.mdone);
    }
  }
  wait_phase(&B.aready, pa++ & 1u, fail);          // head
  tc_fence_after();
#pragma unroll 1
  for (int q = 0; q < kHeadChunks; ++q)
    mma_chunk<128>(a, c, B, f, kColU, kColA + 16u * (uint32_t)q, kAlo, q == 0, fail);
  umma_commit(&B.mdone);
  // every issued MMA done, every requested chunk landed (all are, unless a wait gave up)
  umma_commit(&B.drain);
  if (!mbar_wait(&B.drain, 0u)) *fail = 1;
  for (int x = f.nwait; x < f.nload; ++x)
    if (!mbar_wait(&B.full[x % kStages], (uint32_t)(x / kStages) & 1u)) *fail = 1;
}

// ------------------------------------------------------------------------------------ row threads

// v[i] = parameter p0 + i with the candidate's one patched (p0 is a multiple of 4).
template <int N>
__device__ __forceinline__ void params_at(const TfmArgs& a, const RowCtx& c, unsigned long long p0,
                                          float (&v)[N]) {
  const float4* p = reinterpret_cast<const float4*>(a.params + p0);
#pragma unroll
  for (int i = 0; i < N / 4; ++i) {
    const float4 x = __ldg(p + i);
    v[4 * i] = x.x;
    v[4 * i + 1] = x.y;
    v[4 * i + 2] = x.z;
    v[4 * i + 3] = x.w;
  }
  if (c.midx - p0 < (unsigned long long)N) {
    const int at = (int)(c.midx - p0);
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (i == at) v[i] = c.mval;
  }
}

template <int W>
__device__ __forceinline__ void tmem_store(uint32_t taddr, const uint32_t (&r)[W]) {
  if constexpr (W == 16) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
                 "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]),
                   "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]),
                   "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
  } else {
    static_assert(W == 8, "8 or 16 columns");
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]),
                   "r"(r[6]), "r"(r[7]) : "memory");
  }
}

// N operand values of this row, scaled, as hi and lo fp16 parts in the columns col .. and col + lo ..,
// two values per column.
template <int N>
__device__ __forceinline__ void store_parts(const RowCtx& c, const float (&v)[N], float scale,
                                            uint32_t col, uint32_t lo_off) {
  uint32_t hi[N / 2], lo[N / 2];
#pragma unroll
  for (int q = 0; q < N / 2; ++q) {
    const float x0 = v[2 * q] * scale, x1 = v[2 * q + 1] * scale;
    const __half2 h = __floats2half2_rn(x0, x1);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn(x0 - f.x, x1 - f.y);
    hi[q] = *reinterpret_cast<const uint32_t*>(&h);
    lo[q] = *reinterpret_cast<const uint32_t*>(&l);
  }
  tmem_store(c.tmem + c.trow + col, hi);
  tmem_store(c.tmem + c.trow + col + lo_off, lo);
}

// This warp's operand stores (and shared-memory reads and writes) before the control thread's next
// MMAs and copies.
__device__ __forceinline__ void publish(uint64_t* bar) {
  tc_publish_operands();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) arrive(bar);
}

__device__ __forceinline__ void ld32(const RowCtx& c, uint32_t col, float (&v)[32]) {
  float a0[16], a1[16];
  tmem_ld16(c.tmem + c.trow + col, a0);
  tmem_ld16(c.tmem + c.trow + col + 16u, a1);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    v[i] = a0[i];
    v[16 + i] = a1[i];
  }
}

// Layer norm of row r (its 32 columns here, statistics over all four parts) as the A operand; the
// normalised value of column `stash` (if it is one of this thread's) to s_acol[r].
__device__ __forceinline__ void ln_to_a(const TfmArgs& a, const Ctx& c, unsigned long long og,
                                        unsigned long long ob, int stash, float* s_part,
                                        float* s_acol) {
  float x[32];
  const float* xr = c.xs + c.r * kXLd + 32 * c.g;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 v = *reinterpret_cast<const float4*>(xr + 4 * i);
    x[4 * i] = v.x;
    x[4 * i + 1] = v.y;
    x[4 * i + 2] = v.z;
    x[4 * i + 3] = v.w;
  }
  float s = 0.0f;
#pragma unroll
  for (int i = 0; i < 32; ++i) s += x[i];
  s_part[c.g * kRows + c.r] = s;
  rows_sync();
  const float mean = (((s_part[c.r] + s_part[kRows + c.r]) + s_part[2 * kRows + c.r]) +
                      s_part[3 * kRows + c.r]) / (float)kD;
  float v = 0.0f;
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    const float e = x[i] - mean;
    v = fmaf(e, e, v);
  }
  s_part[(4 + c.g) * kRows + c.r] = v;
  rows_sync();
  const float var = (((s_part[4 * kRows + c.r] + s_part[5 * kRows + c.r]) +
                      s_part[6 * kRows + c.r]) + s_part[7 * kRows + c.r]) / (float)kD;
  const float rstd = rsqrtf(var + a.eps);
  {
    float p[32];
    params_at<32>(a, c, og + 32ull * c.g, p);
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = (x[i] - mean) * rstd * p[i];
    params_at<32>(a, c, ob + 32ull * c.g, p);
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] += p[i];
  }
  if (stash >= 32 * c.g && stash < 32 * c.g + 32) {
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if (32 * c.g + i == stash) s_acol[c.r] = x[i];
  }
  store_parts<32>(c, x, a.f16_ln, kColA + 16u * (uint32_t)c.g, kAlo);
}

template <int MODE>
__global__ void __launch_bounds__(kThreads, 1) tfm_f16_kernel(const __grid_constant__ TfmArgs a) {
  extern __shared__ __align__(1024) unsigned char tsm[];
  __shared__ DeepCand s_c;
  __shared__ int s_tok[2][kT + 1];
  __shared__ float s_part[8 * kRows];
  __shared__ float s_acol[kRows];
  __shared__ float s_zy[kRows];
  __shared__ float s_rowv[kRows];
  __shared__ int s_stage[kKmax];
  __shared__ __align__(8) Bars s_bars;
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail, s_k;
  __shared__ int s_skip[2];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (MODE == kTfmCommit && a.ctl->kstar < a.nscr) return;   // none accepted, or one with a slot
  int k = 0, pair = blockIdx.x;
  if (MODE == kTfmEval) {
    // longest recomputations first: the linear block index is mapped to (candidate rank, sequence
    // pair) with the candidates ranked by the stage they feed, ties by index
    const int Kb = gridDim.x, npair = gridDim.y;
    const int lid = blockIdx.x + blockIdx.y * gridDim.x;
    const int rank = lid / npair;
    pair = lid - rank * npair;
    if (tid < Kb) s_stage[tid] = candidate_stage(a, tid);
    __syncthreads();
    if (tid < Kb) {
      const int my = s_stage[tid];
      int rk = 0;
      for (int q = 0; q < Kb; ++q) rk += (s_stage[q] < my || (s_stage[q] == my && q < tid)) ? 1 : 0;
      if (rk == rank) s_k = tid;
    }
    __syncthreads();
    k = s_k;
  }
  const int s0 = 2 * pair;
  if (tid == 0) {
    if (MODE == kTfmEval) {
      s_c = tfm_candidate(a, k);
    } else if (MODE == kTfmCommit) {
      s_c = a.ctl->acc;
    } else {
      DeepCand d;
      d.idx = 0xffffffffu;
      d.layer = -1;
      d.row = -1;
      d.col = 0;
      d.oldw = d.neww = 0.0f;
      d.delta = 1.0f;
      d.new_code = 0;
      d.valid = 1;
      s_c = d;
    }
    s_fail = 0;
  }
  for (int e = tid; e < 2 * (kT + 1); e += kThreads)
    s_tok[e / (kT + 1)][e % (kT + 1)] = a.tokens[(size_t)s0 * (kT + 1) + e];
  __syncthreads();
  const DeepCand cd = s_c;
  float* part = a.partial + (size_t)k * a.B + s0;
  if (MODE == kTfmEval && k >= tfm_batch_width(a, tfm_batch_tau(a))) {   // past the run's end
    if (tid < 2) part[tid] = 0.0f;
    return;
  }
  // where the recomputed residual streams and sequence losses go: the handle's (commit, forward)
  // or, in an evaluation, the candidate's scratch slot when it has one
  const size_t seq_floats = (size_t)kT * kD;
  const bool slot = MODE == kTfmEval && k < a.nscr;
  float* const xout = MODE != kTfmEval ? a.X
                      : slot ? a.scrX + (size_t)k * (size_t)(2 * a.nL + 1) * a.B * seq_floats
                             : nullptr;
  float* const xmout = MODE != kTfmEval ? a.Xmid
                       : slot ? xout + (size_t)(a.nL + 1) * a.B * seq_floats : nullptr;
  float* const lout = MODE != kTfmEval ? a.ell : slot ? a.scr_ell + (size_t)k * a.B : nullptr;
  if (!cd.valid || cd.delta == 0.0f) {
    if (MODE == kTfmEval && tid < 2) part[tid] = 0.0f;
    return;
  }
  if (tid < 2) {                 // a tok_emb entry: a sequence without that token is unchanged
    int skip = 0;
    if (MODE != kTfmForward && cd.row >= 0) {
      skip = 1;
      for (int t = 0; t < kT; ++t) skip &= s_tok[tid][t] != cd.row;
    }
    s_skip[tid] = skip;
  }
  __syncthreads();
  if (s_skip[0] && s_skip[1]) {
    if (MODE == kTfmEval && tid < 2) part[tid] = 0.0f;
    return;
  }
  const bool fwd = MODE == kTfmForward;
  Ctx c;
  c.g = (warp >> 2) & 3;
  c.r = (warp & 3) * 32 + lane;
  c.sl = c.r / kT;
  c.t = c.r % kT;
  c.trow = (uint32_t)((warp & 3) * 32) << 16;
  c.xs = reinterpret_cast<float*>(tsm);
  c.ring = tsm + kXsBytes;
  c.ks = reinterpret_cast<float*>(c.ring);
  c.vs = c.ks + kRows * kD;
  c.midx = fwd ? ~0ull : (unsigned long long)cd.idx;
  c.mval = cd.neww;
  c.dlt = fwd ? 0.0f : cd.delta;
  c.cstage = fwd ? -1 : cd.layer;
  if (fwd) {
    c.tg.mat = kTcMatNone;
    c.tg.row = c.tg.col = 0;
  } else {
    c.tg = tc_target(a, cd.idx, cd.layer);
  }
  const int b0 = (fwd || cd.layer < 0) ? -1 : cd.layer;
  const int rs = fwd ? kRestartBlock : tfm_restart(a, cd.idx, cd.layer);
  c.unit0 = rs == kRestartUnit;
  c.b0s = b0 < 0 ? 0 : b0 + (c.unit0 ? 1 : 0);
  c.nb = a.nL - c.b0s;
  c.cpb = tfm_f16_block_chunks(a.F);
  c.ffn0 = rs == kRestartFfn;
  c.q0 = c.ffn0 ? kAttnChunks : 0;
  c.total = c.nb * c.cpb - c.q0 + kHeadChunks;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;"
                 ::"r"(smem_u32(&s_tmem)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  Bars& B = s_bars;
  if (tid == 0) {
    for (int q = 0; q < kStages; ++q) {
      mbar_init(&B.full[q], 1);
      mbar_init(&B.empty[q], 1);
    }
    mbar_init(&B.aready, kTfmWorkers / 32);
    mbar_init(&B.mdone, 1);
    mbar_init(&B.drain, 1);
    for (int q = 0; q < 2; ++q) {
      mbar_init(&B.ufull[q], 1);
      mbar_init(&B.a2full[q], kTfmWorkers / 32);
      mbar_init(&B.a2empty[q], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  c.tmem = s_tmem;
  volatile int* fail = &s_fail;

  if (warp == kCtlWarp) {
    if (elect_one()) control(a, c, B, fail);
    __syncwarp();
  } else {
    const float dln = a.f16_dln, dact = a.f16_dact;           // scales of the products
    uint32_t pm = 0u;            // phases of mdone
    int gh = 0;                  // halves of all feed-forward networks so far
    const int nh = a.F / kHc;
    auto product_done = [&]() {
      wait_phase(&B.mdone, pm++ & 1u, fail);
      tc_fence_after();
    };
    auto save = [&](float* base, size_t stream, const float* xr) {   // this row's part of a stream
      float* dst = base + (stream * a.B + s0 + c.sl) * seq_floats + (size_t)c.t * kD + 32 * c.g;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        reinterpret_cast<float4*>(dst)[i] = *reinterpret_cast<const float4*>(xr + 4 * i);
    };
    // residual stream entering the first stage run
    float* xr = c.xs + c.r * kXLd + 32 * c.g;
    if (b0 < 0) {
      const int tok = s_tok[c.sl][c.t];
      float p[32], e[32];
      params_at<32>(a, c, a.o_tok + (unsigned long long)tok * kD + 32 * c.g, p);
      params_at<32>(a, c, a.o_pos + (unsigned long long)c.t * kD + 32 * c.g, e);
#pragma unroll
      for (int i = 0; i < 32; ++i) xr[i] = p[i] + e[i];
      if (xout && !s_skip[c.sl]) save(xout, 0, xr);
    } else if (c.unit0) {
      ffn_unit(a, c, cd, s0, xr, s_part, s_acol);
      if (xout) save(xout, (size_t)(b0 + 1), xr);     // block b0's new output stream
    } else {
      const float* src = (c.ffn0 ? a.Xmid : a.X) + ((size_t)b0 * a.B + s0 + c.sl) * seq_floats +
                         (size_t)c.t * kD + 32 * c.g;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        *reinterpret_cast<float4*>(xr + 4 * i) = reinterpret_cast<const float4*>(src)[i];
    }

#pragma unroll 1
    for (int b = c.b0s; b < a.nL; ++b) {
      const bool here = b == c.cstage;
      const unsigned long long base = a.o_blk0 + (unsigned long long)b * a.blk_size;
      if (!(c.ffn0 && b == c.b0s)) {
        // ---- attention: LN1, Q K V, attention, output projection
        ln_to_a(a, c, base + a.r_ln1g, base + a.r_ln1b,
                (here && c.tg.mat >= kTcQ && c.tg.mat <= kTcV) ? c.tg.col : -1, s_part, s_acol);
        publish(&B.aready);
        rows_sync();               // s_acol complete
        product_done();
        float q[32];
        {
          float v[32], p[32];
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            ld32(c, (m ? kColV : kColK) + 32u * (uint32_t)c.g, v);
            params_at<32>(a, c, base + (m ? a.r_bv : a.r_bk) + 32 * c.g, p);
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = fmaf(v[i], dln, p[i]);
            if (here && c.tg.mat == (m ? kTcV : kTcK))
              add_at(v, c.tg.row - 32 * c.g, c.dlt * s_acol[c.r]);
            float* dst = (m ? c.vs : c.ks) + (size_t)c.r * kD + 32 * c.g;
#pragma unroll
            for (int i = 0; i < 8; ++i)
              *reinterpret_cast<float4*>(dst + 4 * (i ^ (c.r & 7))) =
                  make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
          }
          ld32(c, kColQ + 32u * (uint32_t)c.g, q);
          params_at<32>(a, c, base + a.r_bq + 32 * c.g, p);
#pragma unroll
          for (int i = 0; i < 32; ++i) q[i] = fmaf(q[i], dln, p[i]);
          if (here && c.tg.mat == kTcQ) add_at(q, c.tg.row - 32 * c.g, c.dlt * s_acol[c.r]);
        }
        rows_sync();               // K and V complete
        {
          float o[32];
          attention(c, q, o);
          if (here && c.tg.mat == kTcO) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (32 * c.g + i == c.tg.col) s_acol[c.r] = o[i];
          }
          store_parts<32>(c, o, a.f16_act, kColA + 16u * (uint32_t)c.g, kAlo);
        }
        publish(&B.aready);        // also: this warp is done with K and V
        rows_sync();
        product_done();
        {
          float v[32], p[32];
          ld32(c, kColU + 32u * (uint32_t)c.g, v);
          params_at<32>(a, c, base + a.r_bo + 32 * c.g, p);
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] *= dact;
          if (here && c.tg.mat == kTcO) add_at(v, c.tg.row - 32 * c.g, c.dlt * s_acol[c.r]);
#pragma unroll
          for (int i = 0; i < 32; ++i) xr[i] += v[i] + p[i];
        }
        if (xmout && !s_skip[c.sl]) save(xmout, (size_t)b, xr);
      }
      // ---- feed-forward network, 64 hidden units (16 per thread) at a time
      ln_to_a(a, c, base + a.r_ln2g, base + a.r_ln2b,
              (here && c.tg.mat == kTcW1) ? c.tg.col : -1, s_part, s_acol);
      publish(&B.aready);
      rows_sync();
#pragma unroll 1
      for (int h = 0; h < nh; ++h, ++gh) {
        const uint32_t u2 = 64u * (uint32_t)(h & 1), ph = (uint32_t)(gh >> 1);
        const int f0 = h * kHc + 16 * c.g;
        float p[16];
        params_at<16>(a, c, base + a.r_b1 + f0, p);
        wait_phase(&B.ufull[h & 1], ph & 1u, fail);
        tc_fence_after();
        float u[16];
        tmem_ld16(c.tmem + c.trow + kColU + u2 + 16u * (uint32_t)c.g, u);
#pragma unroll
        for (int i = 0; i < 16; ++i) u[i] *= dln;
        if (here && c.tg.mat == kTcW1) add_at(u, c.tg.row - f0, c.dlt * s_acol[c.r]);
        if (a.act == MCA_ACT_GELU) {
#pragma unroll
          for (int i = 0; i < 16; ++i) u[i] = act_rt(MCA_ACT_GELU, u[i] + p[i], a.g);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) u[i] = act_rt(MCA_ACT_GAUSSIAN, u[i] + p[i], a.g);
        }
        if (here && c.tg.mat == kTcW2) {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (f0 + i == c.tg.col) s_acol[c.r] = u[i];
        }
        if (ph > 0u) {             // the MMAs that read this half's operand columns before
          wait_phase(&B.a2empty[h & 1], (ph - 1u) & 1u, fail);
          tc_fence_after();
        }
        store_parts<16>(c, u, a.f16_act, kColA2 + u2 + 8u * (uint32_t)c.g, kA2lo);
        publish(&B.a2full[h & 1]);
      }
      product_done();
      rows_sync();                 // s_acol complete
      {
        float v[32], p[32];
        ld32(c, kColF + 32u * (uint32_t)c.g, v);
        params_at<32>(a, c, base + a.r_b2 + 32 * c.g, p);
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] *= dact;
        if (here && c.tg.mat == kTcW2) add_at(v, c.tg.row - 32 * c.g, c.dlt * s_acol[c.r]);
#pragma unroll
        for (int i = 0; i < 32; ++i) xr[i] += v[i] + p[i];
      }
      if (xout && !s_skip[c.sl]) save(xout, (size_t)(b + 1), xr);
    }

    // ---- final layer norm, head, next-token cross-entropy
    {
      const bool here = c.cstage == a.nL;
      ln_to_a(a, c, a.o_lnf_g, a.o_lnf_b, (here && c.tg.mat == kTcHead) ? c.tg.col : -1, s_part,
              s_acol);
      publish(&B.aready);
      rows_sync();
      product_done();
      float z[32];
      ld32(c, kColU + 32u * (uint32_t)c.g, z);
#pragma unroll
      for (int i = 0; i < 32; ++i) z[i] *= dln;
      if (here && c.tg.mat == kTcHead) add_at(z, c.tg.row - 32 * c.g, c.dlt * s_acol[c.r]);
      float zmax = -INFINITY;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const int col = 32 * c.g + i;
        z[i] = col < a.V ? z[i] + prm(a, a.o_bh + (unsigned long long)col, c.midx, c.mval)
                         : -INFINITY;
        zmax = fmaxf(zmax, z[i]);
      }
      s_part[c.g * kRows + c.r] = zmax;
      rows_sync();
      const float m = fmaxf(fmaxf(fmaxf(s_part[c.r], s_part[kRows + c.r]), s_part[2 * kRows + c.r]),
                            s_part[3 * kRows + c.r]);
      float se = 0.0f;
      const int y = s_tok[c.sl][c.t + 1];
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        if (32 * c.g + i < a.V) se += exp_fast(z[i] - m);
        if (32 * c.g + i == y) s_zy[c.r] = z[i];
      }
      s_part[(4 + c.g) * kRows + c.r] = se;
      rows_sync();
      if (c.g == 0) {
        const float sum = ((s_part[4 * kRows + c.r] + s_part[5 * kRows + c.r]) +
                           s_part[6 * kRows + c.r]) + s_part[7 * kRows + c.r];
        s_rowv[c.r] = (__logf(sum) + m) - s_zy[c.r];
      }
      rows_sync();
      if (tid < 2) {
        float l = 0.0f;
        for (int t = 0; t < kT; ++t) l += s_rowv[tid * kT + t];
        if (MODE == kTfmEval) part[tid] = s_skip[tid] ? 0.0f : l - a.ell[s0 + tid];
        if (lout && !s_skip[tid]) lout[s0 + tid] = l;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(c.tmem));
  if (tid == 0 && s_fail) atomicCAS(&a.st->err, 0, (int)MCA_ERR_TIMEOUT);
}

// Every weight matrix's image (head rows past the vocabulary are zero). blockIdx.y = 6 b + matrix (Wq,
// Wk, Wv, Wo, W1, W2) or 6 nL for the head.
__global__ void tfm_f16_split_kernel(TfmArgs a) {
  const int slot = blockIdx.y;
  int mat, b = 0, rows = kD, cols = kD;
  unsigned long long src;
  if (slot == 6 * a.nL) {
    mat = kTcHead;
    src = a.o_wh;
  } else {
    b = slot / 6;
    mat = slot % 6;
    const unsigned long long base = a.o_blk0 + (unsigned long long)b * a.blk_size;
    const unsigned int off[6] = {a.r_wq, a.r_wk, a.r_wv, a.r_wo, a.r_w1, a.r_w2};
    src = base + off[mat];
    if (mat == kTcW1) rows = a.F;
    if (mat == kTcW2) cols = a.F;
  }
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < rows * cols; e += gridDim.x * blockDim.x) {
    const int r = e / cols, kk = e - r * cols;
    const float w = (mat == kTcHead && r >= a.V) ? 0.0f : a.params[src + (unsigned long long)e];
    tfm_f16_image_store(a, mat, b, r, kk, w);
  }
}

// Are some of the operands so far below their scales that fp16 parts hold fewer bits than tf32 parts? One
// warp per row of a weight matrix (blockIdx.y as in tfm_f16_split_kernel): the absolute error of its parts is
// 2^-40 q, below 2^-26 of the row's largest weight from 2^-14 q on. The last x block of Wv and of W1
// compares the bound of the activations that it produces with the one that their scale follows from: typical
// ones lie about 2^-9 below their bound and keep 22 bits down to 2^-17 below the scale's.
__global__ void __launch_bounds__(256) tfm_f16_range_kernel(TfmArgs a, float q, float bound, int* out) {
  const int slot = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = slot / 6, mat = slot == 6 * a.nL ? (int)kTcHead : slot % 6;
  const unsigned long long base = a.o_blk0 + (unsigned long long)b * a.blk_size;
  const unsigned int off[6] = {a.r_wq, a.r_wk, a.r_wv, a.r_wo, a.r_w1, a.r_w2};
  const float* w = a.params + (mat == kTcHead ? a.o_wh : base + off[mat]);
  const int rows = mat == kTcHead ? a.V : mat == kTcW1 ? a.F : kD;
  const int cols = mat == kTcW2 ? a.F : kD;
  if (blockIdx.x + 1 < gridDim.x) {
    for (int r = blockIdx.x * 8 + warp; r < rows; r += 8 * (gridDim.x - 1)) {
      float m = 0.0f;
      for (int k = lane; k < cols; k += 32) m = fmaxf(m, fabsf(w[(size_t)r * cols + k]));
      m = __int_as_float(__reduce_max_sync(0xffffffffu, __float_as_int(m)));
      if (lane == 0 && m > 0.0f && m < q * 0x1p-14f) *out = 1;
    }
    return;
  }
  if (mat != kTcV && mat != kTcW1) return;
  __shared__ int s_m[3];                // bits of the largest weight, layer-norm gain or bias, own bias
  if (threadIdx.x < 3) s_m[threadIdx.x] = 0;
  __syncthreads();
  const float* ln = a.params + base + (mat == kTcV ? a.r_ln1g : a.r_ln2g);
  const float* lb = a.params + base + (mat == kTcV ? a.r_ln1b : a.r_ln2b);
  const float* bi = a.params + base + (mat == kTcV ? a.r_bv : a.r_b1);
  int m[3] = {0, 0, 0};
  for (int e = threadIdx.x; e < rows * cols; e += 256) m[0] = max(m[0], __float_as_int(fabsf(w[e])));
  for (int e = threadIdx.x; e < kD; e += 256)
    m[1] = max(m[1], __float_as_int(fmaxf(fabsf(ln[e]), fabsf(lb[e]))));
  for (int e = threadIdx.x; e < rows; e += 256) m[2] = max(m[2], __float_as_int(fabsf(bi[e])));
  for (int i = 0; i < 3; ++i) {
    m[i] = __reduce_max_sync(0xffffffffu, m[i]);
    if (lane == 0) atomicMax(&s_m[i], m[i]);
  }
  __syncthreads();
  if (threadIdx.x == 0 && 256.0f * __int_as_float(s_m[1]) * __int_as_float(s_m[0]) +
                                  __int_as_float(s_m[2]) < bound * 0x1p-8f)
    *out = 1;
}

template <int MODE>
cudaError_t launch_f16(const TfmArgs& a, dim3 grid, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute((const void*)tfm_f16_kernel<MODE>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return e;
  tfm_f16_kernel<MODE><<<grid, kThreads, kSmem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_tfm_f16_split(const TfmArgs& a, cudaStream_t s) {
  tfm_f16_split_kernel<<<dim3(32, 6 * a.nL + 1), 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_tfm_f16_range(const TfmArgs& a, float q, float bound, int* out, cudaStream_t s) {
  tfm_f16_range_kernel<<<dim3(17, 6 * a.nL + 1), 256, 0, s>>>(a, q, bound, out);
  return cudaGetLastError();
}

cudaError_t launch_tfm_f16(const TfmArgs& a, int mode, cudaStream_t s) {
  const int Kb = a.n_explicit > 0 ? a.n_explicit : a.Kb;
  if (mode == kTfmEval) return launch_f16<kTfmEval>(a, dim3(Kb, a.B / 2), s);
  if (mode == kTfmCommit) return launch_f16<kTfmCommit>(a, dim3(a.B / 2), s);
  return launch_f16<kTfmForward>(a, dim3(a.B / 2), s);
}

}  // namespace mca

// Deep MLP path on the 5th-generation tensor cores: the dense part of a candidate's chain,
//   Z'_m = Z_m + W_m (f(Z'_{m-1}) - f(Z_{m-1})),   m = l+2 .. L-2   (Section 2.4),
// as error-compensated three-product tcgen05 MMAs with the accumulator in tensor memory.
//
// One CTA per (candidate, tile of kTcTS = 128 samples): 16 worker warps and one control warp. Per
// dense layer the CTA computes the transposed change D^T[samples x 256] = A[samples x 256] W_m^T,
// where A holds the previous layer's activation changes split as A = A_hi + A_lo and W_m = W_hi + W_lo
// (kept split in global memory, updated with every commit), each part with an 11-bit significand:
//   D = A_lo W_hi^T + A_hi W_lo^T + A_hi W_hi^T      (the A_lo W_lo^T term, ~2^-22 relative, dropped)
// Tanh layers use fp16 parts (kind::f16, K = 16 per MMA): |change| <= 2 and the largest weight's
// magnitude are scaled by powers of two to at most 2^15, so that an element x is represented to 2^-22 of
// itself or 2^-40 of the largest, whichever is larger, and D is scaled back exactly. Weights of which
// too many lie that far below the largest (deep_wide_kernel), layers whose
// changes have no bound (ReLU, GELU, identity) or another function use tf32 parts (K = 8 per MMA,
// the same time per MMA, hence half the rate).
//
// The layers are pipelined chunk by chunk. The workers produce A in K chunks (32 fp16 or 16 tf32
// features; hi and lo, 16 KB) into a ring of four shared-memory slots; the control thread issues each
// chunk's six MMAs as soon as the chunk and its weight stage are there, so layer m+1's MMAs run while
// the workers are still forming layer m's later chunks. Two accumulators in tensor memory (columns
// [0, 256) and [256, 512)) alternate by layer: the workers read layer m's finished D while the
// MMAs of layer m+1 fill the other one. W streams through four 32 KB stages (one chunk, hi + lo),
// each one bulk copy, reaching across layer boundaries. All operands are K-major without swizzle:
// 8-row x 16-byte core matrices. One elected thread of the converged control warp issues the MMAs.
// 24 layers of 256 on 10000 samples, about two candidates per batch: 400 us per batch with tf32 parts,
// two exponentials and two reciprocals per element and 16 features a step; 259 us with fp16 parts,
// one reciprocal and 32 features a step.
//
// Worker warp w reads tensor-memory lanes 32 (w mod 4) .. + 31 (its samples) and, in every chunk,
// one quarter of the features (part w / 4): the cached field + D gives the new field, the next activation
// change f(z') - f(z) (exactly 0 where a field did not change) goes into the ring, and after the
// last dense layer the changes accumulate into the output layer instead. Every per-(candidate,
// tile) loss change depends only on that pair: the trajectory does not depend on the batch width.
// COMMIT writes the fields exactly as the evaluation computed them. Every wait is bounded (2 s); on a
// time-out the CTA records MCA_ERR_TIMEOUT, lets its issued copies and MMAs complete (bounded) and
// frees its tensor memory.
#include <cuda_fp16.h>

#include "mca_deep.cuh"
#include "mca_device.cuh"
#include "mca_internal.h"
#include "mca_tc.cuh"

namespace mca {
namespace {

constexpr int kWorkWarps = 16;
constexpr int kTcThreads = (kWorkWarps + 1) * 32;   // + one control warp
constexpr int kCtl = kWorkWarps * 32;                // the control thread
constexpr int kParts = 4;                            // feature parts per lane quarter
constexpr int kTcW = 256;                            // width of the dense layers
constexpr int kChunkBytes = 64;                      // K chunk of one row: 16 tf32 or 32 fp16
constexpr int kAHalf = kTcTS * kChunkBytes;          // 8 KB: hi or lo of one A chunk
constexpr int kASlot = 2 * kAHalf;
constexpr int kASlots = 4;
constexpr int kWHalfBytes = kTcW * kChunkBytes;      // 16 KB: hi or lo of one W chunk
constexpr int kWStageBytes = 2 * kWHalfBytes;        // 32 KB
constexpr int kStages = 4;
constexpr int kTcSmem = kASlots * kASlot + kStages * kWStageBytes;
// core-matrix strides (bytes): A chunk: K groups 2 KB apart, sample groups 128 B apart;
// W stage: K groups 4 KB apart, row groups 128 B apart. The split weights of a layer are kept in
// global memory as consecutive 32 KB stage images, one per chunk (hi then lo), so that one bulk copy
// fills a stage.
constexpr uint32_t kALBO = (kTcTS / 8) * 128, kASBO = 128;
constexpr uint32_t kWLBO = (kTcW / 8) * 128, kWSBO = 128;

// The operand split (see the head of this file). kKC: features per chunk; kNQ: those of one worker
// thread (one 16-byte core-matrix row); M = 128, N = 256, D fp32, operands K-major.
template <bool F16>
struct Split;
template <>
struct Split<false> {
  static constexpr int kKC = 16, kNQ = 4;
  static constexpr uint32_t kIdesc = tc_idesc_tf32(kTcTS, kTcW);
};
template <>
struct Split<true> {
  static constexpr int kKC = 32, kNQ = 8;
  static constexpr uint32_t kIdesc = tc_idesc_f16(kTcTS, kTcW);
};

static_assert(kTcSmem + 2048 <= 227 * 1024, "shared memory of the chain kernel");
static_assert((kParts - 1) * kMaxC * kTcTS * 4 <= kStages * kWStageBytes, "output scratch");

// One thread: stage st <- the 32 KB image of one chunk, completion counted on mbarrier full.
__device__ __forceinline__ void load_stage(uint32_t dst, const void* src, uint64_t* full) {
  bulk_load(dst, src, (uint32_t)kWStageBytes, full);
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Field rows of one layer for this tile into L2: worker thread t, row t / 2, two 128-byte lines.
__device__ __forceinline__ void prefetch_tile(const float* Zm, int Np, int n0, int t) {
  const float* r = Zm + (size_t)(t >> 1) * Np + n0 + 64 * (t & 1);
  prefetch_l2(r);
  prefetch_l2(r + 32);
}

// N (4 or 8) accumulator columns of this thread's lane into r, left in flight: the values may be read
// only after tmem_wait(r).
__device__ __forceinline__ void tmem_issue(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_issue(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}

// Wait for this thread's tensor-memory loads; r is tied to the wait so that no read of it moves
// above it.
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]) :: "memory");
}
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                 "+r"(r[6]), "+r"(r[7]) :: "memory");
}

// Every lane waits for the phase; true in every lane iff no lane timed out.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity) ? 1 : 0) != 0;
}

// x (two values) as fp16 hi and lo parts.
__device__ __forceinline__ void split_f16x2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(x0, x1);
  const float2 f = __half22float2(h);
  const __half2 l = __floats2half2_rn(x0 - f.x, x1 - f.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// Worker: put the activation changes d of sample s (part fp of the chunk's features) into ring slot
// ga % kASlots as hi and lo parts, once the MMAs of the chunk kASlots earlier are done with the slot;
// then the warp's arrival on the slot's full barrier.
template <bool F16, int NQ>
__device__ __forceinline__ bool produce_chunk(unsigned char* aring, uint64_t* afull,
                                              uint64_t* aempty, int ga, int fp, int s,
                                              const float (&d)[NQ]) {
  const int as = ga % kASlots;
  if (ga >= kASlots && !warp_wait(&aempty[as], (uint32_t)((ga / kASlots) - 1) & 1u)) return false;
  unsigned char* slot = aring + (size_t)as * kASlot + (size_t)fp * kALBO + (size_t)s * 16;
  if constexpr (F16) {
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) split_f16x2(d[2 * q], d[2 * q + 1], hi[q], lo[q]);
    *reinterpret_cast<uint4*>(slot) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(slot + kAHalf) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  } else {
    float hi[4], lo[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      hi[q] = tf32_rna(d[q]);
      lo[q] = tf32_rna(d[q] - hi[q]);
    }
    *reinterpret_cast<float4*>(slot) = make_float4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<float4*>(slot + kAHalf) = make_float4(lo[0], lo[1], lo[2], lo[3]);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncwarp();
  if ((threadIdx.x & 31) == 0)
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&afull[as])) : "memory");
  return true;
}

// e^{2z}, z cut at 20 from above.
__device__ __forceinline__ float exp2z(float z) {
  float m;
  asm("min.NaN.f32 %0, %1, 0f41A00000;" : "=f"(m) : "f"(z));
  return ex2_ftz(m * (2.0f * kLog2e));
}

// Change of one hidden activation. F16 (tanh layers): kDeepDScale (tanh(zn) - tanh(zo)), exactly 0 when
// zn == zo, from u = e^{2z} as 2 (un - uo) / ((un + 1)(uo + 1)): three of the special-function unit's
// operations instead of four, and no cancellation between two rounded tanh values. z is cut at 20
// (tanh = 1 to 2e-17) so that the product stays finite; a NaN stays a NaN.
template <int ACTH, bool F16>
__device__ __forceinline__ float act_change(float zn, float zo, float g, int act_rt_) {
  if constexpr (F16) {
    const float un = exp2z(zn), uo = exp2z(zo);
    const float t = uo + 1.0f;
    return (un - uo) * rcp_ftz(fmaf(un, t, t)) * (2.0f * kDeepDScale);
  } else {
    return zn != zo ? act<ACTH>(zn, g, act_rt_) - act<ACTH>(zo, g, act_rt_) : 0.0f;
  }
}

// MODE: evaluation of a candidate, its commit, or the forward pass from Z_0 on (every later field and the
// losses; the chain's "changes" are then the activations themselves). ACTH: transfer function of the
// hidden layers (-1: read per layer at run time).
enum ChainMode { kChainEval = 0, kChainCommit = 1, kChainForward = 2 };

template <int MODE, int ACTH, bool F16>
__global__ void __launch_bounds__(kTcThreads, 1) deep_chain_tc_kernel(DeepArgs a) {
  constexpr int kKC = Split<F16>::kKC, NQ = Split<F16>::kNQ, kChunks = kTcW / kKC;
  constexpr uint32_t kIdesc = Split<F16>::kIdesc;
  constexpr bool COMMIT = MODE == kChainCommit, FWD = MODE == kChainForward;
  extern __shared__ __align__(1024) unsigned char tsm[];
  unsigned char* aring = tsm;                                 // A chunks
  unsigned char* wst = tsm + kASlots * kASlot;                // W stages
  __shared__ DeepCand s_cand;
  __shared__ float s_da[kTcTS];
  __shared__ float s_red[32];
  __shared__ __align__(8) uint64_t s_wfull[kStages], s_wempty[kStages];
  __shared__ __align__(8) uint64_t s_afull[kASlots], s_aempty[kASlots];
  __shared__ __align__(8) uint64_t s_dfull[2], s_drain;
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_fail;
  __shared__ int s_k;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int k = 0, tile = MODE != kChainEval ? blockIdx.x : 0;
  if (COMMIT && a.ctl->kstar < 0) return;
  if (MODE == kChainEval) {
    // Longest chains first: CTAs start in linear block order, so the linear index is mapped to
    // (candidate rank, tile) with the candidates ranked by the depth of their dense chain (the
    // mutated layer, from the proposal alone), ties by index. Every CTA computes the same ranking.
    const int Kb = gridDim.x;
    const int lid = blockIdx.x + blockIdx.y * gridDim.x;
    const int rank = lid / a.ntiles;
    tile = lid - rank * a.ntiles;
    if (tid < Kb) {
      const int my = deep_candidate_layer(a, tid);
      int rk = 0;
      for (int q = 0; q < Kb; ++q) {
        const int lq = deep_candidate_layer(a, q);
        rk += (lq < my || (lq == my && q < tid)) ? 1 : 0;     // shallower layer = longer chain
      }
      if (rk == rank) s_k = tid;
    }
    __syncthreads();
    k = s_k;
  }
  const int n0 = tile * kTcTS;
  if (tid == 0) {
    if (FWD) {                       // the dense chain starts at layer 1
      s_cand = DeepCand{0u, -1, 0, 0, 0.0f, 0.0f, 1.0f, 0, 1};
    } else {
      s_cand = COMMIT ? a.ctl->acc : deep_candidate(a, k);
    }
    s_fail = 0;
  }
  __syncthreads();
  const DeepCand c = s_cand;
  float* part = a.partial + (size_t)k * a.ntiles + tile;
  if (!FWD && (!c.valid || c.delta == 0.0f)) {
    if (!COMMIT && tid == 0) *part = 0.0f;
    return;
  }
  const int L = a.L, l = c.layer, j = c.row, i = c.col;
  const int Np = a.Np, N = a.N;
  float dl = 0.0f;
  // this candidate's scratch slot, when it has one and a dense chain (layer <= L-3)
  float* const* sk = (MODE == kChainEval && k < a.nscr && l <= L - 3) ? a.scr + (size_t)k * (L + 1) : nullptr;
  if (l + 1 < L - 1 && a.n_out[l + 1] == kTcW && tid < kCtl) prefetch_tile(a.Z[l + 1], Np, n0, tid);

  // ---- row j of layer l (thread s = sample)
  if (!FWD && tid < kTcTS) {
    const int n = n0 + tid;
    float da = 0.0f;
    if (n < N) {
      const float v = l == 0 ? a.XT[(size_t)i * Np + n]
                             : act_rt(a.act[l - 1], a.Z[l - 1][(size_t)i * Np + n], a.g[l - 1]);
      float* zp = a.Z[l] + (size_t)j * Np + n;
      const float z = *zp;
      const float zn = fmaf(c.delta, v, z);
      if (l == L - 1) {                              // an output weight: output field j changes
        float zz[kMaxC];
#pragma unroll
        for (int q = 0; q < kMaxC; ++q)
          zz[q] = q < a.C ? a.Z[l][(size_t)q * Np + n] : 0.0f;
#pragma unroll
        for (int q = 0; q < kMaxC; ++q)
          if (q == j) zz[q] = zn;
        dl = out_delta<COMMIT>(a, n, zz, zn != z);
      } else {
        da = act_rt(a.act[l], zn, a.g[l]) - act_rt(a.act[l], z, a.g[l]);
        if (COMMIT) *zp = zn;
        if (sk) sk[l][(size_t)j * Np + n] = zn;
      }
    }
    s_da[tid] = da;
  }
  __syncthreads();

  if (l == L - 2) {
    // ---- layer l+1 is the output layer: rank-1 change of the output fields
    if (tid < kTcTS) {
      const int n = n0 + tid;
      const float da = s_da[tid];
      const float* W1 = a.w[L - 1];
      if (n < N && da != 0.0f) {
        float zz[kMaxC];
        bool changed = false;
#pragma unroll
        for (int q = 0; q < kMaxC; ++q) {
          if (q < a.C) {
            const float zo = a.Z[L - 1][(size_t)q * Np + n];
            zz[q] = fmaf(W1[(size_t)q * a.n_in[L - 1] + j], da, zo);
            changed |= zz[q] != zo;
          } else {
            zz[q] = 0.0f;
          }
        }
        dl = out_delta<COMMIT>(a, n, zz, changed);
      }
    }
  } else if (l < L - 2) {
    const bool dense = l + 2 <= L - 2;
    const int nd = dense ? (L - 2) - (l + 2) + 1 : 0;      // dense layers of the chain
    const int nchunks = nd * kChunks;
    const bool worker = warp < kWorkWarps;
    const int qd = warp & 3, fp = (warp >> 2) & 3;        // lane quarter, feature part
    const int s = qd * 32 + lane, n = n0 + s;
    const bool live = worker && n < N;
    const uint32_t lane_base = (uint32_t)(qd * 32) << 16;
    uint32_t tmem = 0;
    if (dense) {
      if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;"
                     ::"r"(smem_u32(&s_tmem)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
      }
      if (tid == kCtl) {
        for (int q = 0; q < kStages; ++q) {
          mbar_init(&s_wfull[q], 1);
          mbar_init(&s_wempty[q], 1);
        }
        for (int q = 0; q < kASlots; ++q) {
          mbar_init(&s_afull[q], kWorkWarps);
          mbar_init(&s_aempty[q], 1);
        }
        mbar_init(&s_dfull[0], 1);
        mbar_init(&s_dfull[1], 1);
        mbar_init(&s_drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // the first weight chunks of the first dense layer load during the rank-1 step
        const unsigned char* w0 = reinterpret_cast<const unsigned char*>(a.whi[l + 2]);
        const uint32_t sw0 = smem_u32(wst);
        for (int q = 0; q < kStages - 1 && q < nchunks; ++q)
          load_stage(sw0 + (uint32_t)(q * kWStageBytes), w0 + (size_t)q * kWStageBytes, &s_wfull[q]);
      }
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      tmem = s_tmem;
    }
    float outp[kMaxC];
#pragma unroll
    for (int q = 0; q < kMaxC; ++q) outp[q] = 0.0f;
    const float* Wout = a.w[L - 1];
    const int Kout = a.n_in[L - 1];
    auto out_add = [&](const float (&d)[NQ], int f0) {   // the output layer's change, features f0 ..
#pragma unroll
      for (int q = 0; q < NQ; ++q)
#pragma unroll
        for (int o = 0; o < kMaxC; ++o)
          if (o < a.C) outp[o] = fmaf(Wout[(size_t)o * Kout + f0 + q], d[q], outp[o]);
    };

    if (!worker) {
      // ---- control warp, one elected thread: every dense layer's MMAs, chunk by chunk as the
      // workers produce A
      if (dense && elect_one()) {
        const uint32_t sw = smem_u32(wst), sa = smem_u32(aring);
        const uint64_t a0 = umma_desc(sa, kALBO, kASBO), w0 = umma_desc(sw, kWLBO, kWSBO);
        int issued_w = kStages - 1 < nchunks ? kStages - 1 : nchunks;   // weight chunks requested
        int landed_w = 0;                                               // ... and waited for
        bool ok = true;
        for (int gc = 0; gc < nchunks && ok; ++gc) {
          const int li = gc / kChunks, cc = gc % kChunks;
          const int as = gc % kASlots, st = gc % kStages;
          if (!mbar_wait(&s_wfull[st], (uint32_t)(gc / kStages) & 1u)) {
            ok = false;
            break;
          }
          landed_w = gc + 1;
          if (!mbar_wait(&s_afull[as], (uint32_t)(gc / kASlots) & 1u)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t dt = tmem + (uint32_t)(li & 1) * 256u;
          // descriptors count 16-byte units
          const uint64_t ab = a0 + (uint64_t)(as * (kASlot / 16));
          const uint64_t wb = w0 + (uint64_t)(st * (kWStageBytes / 16));
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) {           // K steps of 8 tf32 / 16 fp16: two K groups each
            const uint64_t dahi = ab + (uint64_t)(ks * 2 * (kALBO / 16));
            const uint64_t dalo = dahi + kAHalf / 16;
            const uint64_t dwhi = wb + (uint64_t)(ks * 2 * (kWLBO / 16));
            const uint64_t dwlo = dwhi + kWHalfBytes / 16;
            const uint32_t first = (cc > 0 || ks > 0) ? 1u : 0u;
            if constexpr (F16) {
              mma_ss_f16(dt, dalo, dwhi, kIdesc, first);
              mma_ss_f16(dt, dahi, dwlo, kIdesc, 1u);
              mma_ss_f16(dt, dahi, dwhi, kIdesc, 1u);
            } else {
              mma_ss(dt, dalo, dwhi, kIdesc, first);
              mma_ss(dt, dahi, dwlo, kIdesc, 1u);
              mma_ss(dt, dahi, dwhi, kIdesc, 1u);
            }
          }
          umma_commit(&s_aempty[as]);
          umma_commit(&s_wempty[st]);
          if (cc == kChunks - 1) umma_commit(&s_dfull[li & 1]);
          // chunk gc + kStages - 1 goes to the stage chunk gc - 1 used, once its MMAs are done
          const int nc = gc + kStages - 1;
          if (nc < nchunks) {
            const int ns = nc % kStages;
            if (gc >= 1 && !mbar_wait(&s_wempty[ns], (uint32_t)((gc - 1) / kStages) & 1u)) {
              ok = false;
              break;
            }
            const int nl = l + 2 + nc / kChunks, nci = nc % kChunks;
            load_stage(sw + (uint32_t)(ns * kWStageBytes),
                       reinterpret_cast<const unsigned char*>(a.whi[nl]) +
                           (size_t)nci * kWStageBytes,
                       &s_wfull[ns]);
            issued_w = nc + 1;
          }
        }
        if (!ok) s_fail = 1;
        // drain: every MMA issued above complete, every requested weight chunk landed
        umma_commit(&s_drain);
        if (!mbar_wait(&s_drain, 0u)) s_fail = 1;
        for (int q = landed_w; q < issued_w; ++q)
          if (!mbar_wait(&s_wfull[q % kStages], (uint32_t)(q / kStages) & 1u)) s_fail = 1;
      }
      __syncwarp();
    } else {
      // ---- workers
      bool ok = true;
      int ga = 0;                                         // A chunks produced
      const float dsc = F16 ? a.tc_dscale : 1.0f;         // the products' scale
      // layer l+1: rank-1 change through column j of W_{l+1}; its activation change is the first
      // A (dense) or feeds the output layer directly (l = L-3)
      if (dense && !FWD) prefetch_tile(a.Z[l + 2], Np, n0, tid);
      {
        const int m1 = l + 1;
        const float* W1 = a.w[m1];
        const int K1 = a.n_in[m1];
        const float da = FWD ? 0.0f : s_da[s];
        float* Zm = a.Z[m1];
        const bool moves = live && da != 0.0f;
        // loads one chunk ahead of their use (n < Np: always in the array)
        float wv[NQ], zo[NQ], wv_n[NQ], zo_n[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          wv_n[q] = FWD ? 0.0f : W1[(size_t)(fp * NQ + q) * K1 + j];
          zo_n[q] = Zm[(size_t)(fp * NQ + q) * Np + n];
        }
#pragma unroll 1
        for (int cc = 0; cc < kChunks; ++cc) {
          const int f0 = cc * kKC + fp * NQ;
          float d[NQ];
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            wv[q] = wv_n[q];
            zo[q] = zo_n[q];
          }
          if (cc + 1 < kChunks) {
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
              wv_n[q] = FWD ? 0.0f : W1[(size_t)(f0 + kKC + q) * K1 + j];
              zo_n[q] = Zm[(size_t)(f0 + kKC + q) * Np + n];
            }
          }
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            if (FWD) {
              d[q] = tanh_exp(zo[q]) * kDeepDScale;
              continue;
            }
            const float zn = moves ? fmaf(wv[q], da, zo[q]) : zo[q];
            d[q] = act_change<ACTH, F16>(zn, zo[q], a.g[m1], a.act[m1]);
            if (COMMIT && zn != zo[q]) Zm[(size_t)(f0 + q) * Np + n] = zn;
            if (sk) sk[m1][(size_t)(f0 + q) * Np + n] = zn;
          }
          if (dense) {
            if (!produce_chunk<F16>(aring, s_afull, s_aempty, ga, fp, s, d)) {
              ok = false;
              break;
            }
            ++ga;
          } else {
            out_add(d, f0);
          }
        }
      }
      // dense layers m = l+2 .. L-2: read D of layer m as its MMAs finish, form the next A
      float zo_n[NQ];                                     // cached fields one chunk ahead
      if (dense) {
#pragma unroll
        for (int q = 0; q < NQ; ++q)
          zo_n[q] = FWD ? 0.0f : a.Z[l + 2][(size_t)(fp * NQ + q) * Np + n];
      }
      for (int li = 0; li < nd && ok; ++li) {
        const int m = l + 2 + li;
        const bool last = m == L - 2;
        if (!last && !FWD) prefetch_tile(a.Z[m + 1], Np, n0, tid);
        if (!warp_wait(&s_dfull[li & 1], (uint32_t)(li >> 1) & 1u)) {
          ok = false;
          break;
        }
        tc_fence_after();
        float* Zm = a.Z[m];
        float* Sm = sk ? sk[m] : nullptr;
        const float* Zn = last ? Zm : a.Z[m + 1];
        const uint32_t dt = tmem + lane_base + (uint32_t)(li & 1) * 256u;
        // accumulator columns one chunk ahead: chunk cc + 1's load is in flight while chunk cc is
        // processed
        uint32_t dr_n[NQ];
        tmem_issue(dt + (uint32_t)(fp * NQ), dr_n);
        tmem_wait(dr_n);
#pragma unroll 1
        for (int cc = 0; cc < kChunks; ++cc) {
          const int f0 = cc * kKC + fp * NQ;
          float zo[NQ], zn[NQ], d[NQ];
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            zo[q] = zo_n[q];
            zn[q] = FWD ? __uint_as_float(dr_n[q]) * dsc
                    : F16 ? fmaf(__uint_as_float(dr_n[q]), dsc, zo[q])
                          : zo[q] + __uint_as_float(dr_n[q]);
          }
          if (cc + 1 < kChunks) tmem_issue(dt + (uint32_t)(f0 + kKC), dr_n);
          if (!FWD) {                          // the next chunk's cached fields, one chunk ahead
            const float* src = cc + 1 < kChunks ? Zm + (size_t)(f0 + kKC) * Np + n
                                                : Zn + (size_t)(fp * NQ) * Np + n;
#pragma unroll
            for (int q = 0; q < NQ; ++q) zo_n[q] = src[(size_t)q * Np];
          }
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            if (FWD) {
              d[q] = tanh_exp(zn[q]) * kDeepDScale;
              Zm[(size_t)(f0 + q) * Np + n] = zn[q];
              continue;
            }
            if (!live) zn[q] = zo[q];
            d[q] = act_change<ACTH, F16>(zn[q], zo[q], a.g[m], a.act[m]);
            if (COMMIT && zn[q] != zo[q]) Zm[(size_t)(f0 + q) * Np + n] = zn[q];
            if (Sm) Sm[(size_t)(f0 + q) * Np + n] = zn[q];
          }
          bool okc = true;
          if (!last) {
            okc = produce_chunk<F16>(aring, s_afull, s_aempty, ga, fp, s, d);
            ++ga;
          } else {
            out_add(d, f0);
          }
          tmem_wait(dr_n);                     // chunk cc + 1's columns (none in flight at the end)
          if (!okc) {
            ok = false;
            break;
          }
        }
      }
      if constexpr (F16) {
#pragma unroll
        for (int o = 0; o < kMaxC; ++o) outp[o] *= 1.0f / kDeepDScale;
      }
      if (!ok) s_fail = 1;
    }

    // ---- output layer: the feature parts of each sample, in a fixed order
    tc_fence_before();
    __syncthreads();                                  // the control thread has drained
    float* xo = reinterpret_cast<float*>(wst);        // W stages are free now
    if (worker && fp >= 1) {
#pragma unroll
      for (int o = 0; o < kMaxC; ++o) xo[((fp - 1) * kMaxC + o) * kTcTS + s] = outp[o];
    }
    __syncthreads();
    if (worker && fp == 0) {
#pragma unroll
      for (int p = 1; p < kParts; ++p)
#pragma unroll
        for (int o = 0; o < kMaxC; ++o) outp[o] += xo[((p - 1) * kMaxC + o) * kTcTS + s];
    }
    const bool failed = s_fail != 0;                  // the same value in every thread here
    if (FWD) {
      if (worker && fp == 0 && !failed) {
        const int Lo = L - 1;
#pragma unroll
        for (int o = 0; o < kMaxC; ++o)
          if (o < a.C) a.Z[Lo][(size_t)o * Np + n] = outp[o];
        if (live)
          a.ell[n] = sample_loss<-1, -1, kMaxC>(outp, a.C, a.y[n], a.g[Lo], a.act[Lo], a.loss);
      }
    } else if (worker && fp == 0 && live && !failed) {
      float zz[kMaxC];
      bool changed = false;
#pragma unroll
      for (int o = 0; o < kMaxC; ++o) {
        if (o < a.C) {
          const float zo = a.Z[L - 1][(size_t)o * Np + n];
          zz[o] = zo + outp[o];
          changed |= zz[o] != zo;
        } else {
          zz[o] = 0.0f;
        }
      }
      dl = out_delta<COMMIT>(a, n, zz, changed);
      if (sk) {                                       // the same output fields and loss as a commit
#pragma unroll
        for (int o = 0; o < kMaxC; ++o)
          if (o < a.C) sk[L - 1][(size_t)o * Np + n] = zz[o];
        const int Lo = L - 1;
        sk[L][n] = changed ? sample_loss<-1, -1, kMaxC>(zz, a.C, a.y[n], a.g[Lo], a.act[Lo], a.loss)
                           : a.ell[n];
      }
    } else if (sk && worker && fp == 0 && !failed) {  // padding samples keep their values
#pragma unroll
      for (int o = 0; o < kMaxC; ++o)
        if (o < a.C) sk[L - 1][(size_t)o * Np + n] = a.Z[L - 1][(size_t)o * Np + n];
      sk[L][n] = a.ell[n];
    }
    if (dense) {
      tc_fence_after();
      if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
      if (tid == 0 && failed) atomicCAS(&a.st->err, 0, (int)MCA_ERR_TIMEOUT);
    }
  }
  if (MODE == kChainEval) {
    const float tot = block_sum(dl, s_red);
    if (tid == 0) *part = tot;
  }
}

// W_hi and W_lo of every dense layer, stored as the stage images the chain kernel copies (chunk c:
// hi then lo, core-matrix order).
__global__ void deep_split_kernel(DeepArgs a) {
  const int m = blockIdx.y + 1;
  if (m > a.L - 2 || a.whi[m] == nullptr) return;
  const int n = kTcW * kTcW;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x)
    deep_tc_image_store(a, m, e / kTcW, e % kTcW, a.w[m][e]);
}

// Row r of dense layer m: the weights, or those behind the masks.
__device__ __forceinline__ const float* dense_row(const DeepArgs& a, int m, int r) {
  return (a.wk[m] == MCA_W_MASKED_FP32 ? a.wfix[m] : a.w[m]) + (size_t)r * kTcW;
}

__global__ void deep_top_kernel(DeepArgs a, int* top) {
  const int m = blockIdx.y + 1, lane = threadIdx.x & 31;
  const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (m > a.L - 2 || r >= kTcW) return;
  const float* w = dense_row(a, m, r);
  int v = 0;                         // the bits of non-negative floats order like the floats
#pragma unroll
  for (int k = lane; k < kTcW; k += 32) v = max(v, __float_as_int(fabsf(w[k])));
  v = __reduce_max_sync(0xffffffffu, v);
  if (lane == 0) atomicMax(top, v);
}

// One warp per row of a dense layer: are more than wide_allowance of its weights below 2^-kWideGap of the
// bound?
__global__ void deep_wide_kernel(DeepArgs a, const int* top, float floor, int* out) {
  const int m = blockIdx.y + 1, lane = threadIdx.x & 31;
  const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (m > a.L - 2 || r >= kTcW) return;
  const float b = fmaxf(floor, top ? __int_as_float(*top) : 0.0f);
  const int limit = (__float_as_int(b) >> 23) + 1 - kWideGap;   // exponents below it
  const float* w = dense_row(a, m, r);
  unsigned int n = 0, low = 0;
#pragma unroll
  for (int k = lane; k < kTcW; k += 32) {
    const float v = fabsf(w[k]);
    n += v != 0.0f;
    low += v != 0.0f && (__float_as_int(v) >> 23) < limit;
  }
  n = __reduce_add_sync(0xffffffffu, n);
  low = __reduce_add_sync(0xffffffffu, low);
  if (lane == 0 && low > wide_allowance(n)) *out = 1;
}

}  // namespace

cudaError_t launch_deep_top(const DeepArgs& a, int* top, cudaStream_t s) {
  deep_top_kernel<<<dim3(kTcW / 8, a.L - 2), 256, 0, s>>>(a, top);
  return cudaGetLastError();
}

cudaError_t launch_deep_wide(const DeepArgs& a, const int* top, float floor, int* out,
                             cudaStream_t s) {
  deep_wide_kernel<<<dim3(kTcW / 8, a.L - 2), 256, 0, s>>>(a, top, floor, out);
  return cudaGetLastError();
}

cudaError_t launch_deep_split(const DeepArgs& a, cudaStream_t s) {
  if (a.L < 3) return cudaSuccess;
  deep_split_kernel<<<dim3(64, a.L - 2), 256, 0, s>>>(a);
  return cudaGetLastError();
}

template <int MODE>
static cudaError_t launch_tc(const DeepArgs& a, dim3 grid, cudaStream_t s) {
  const void* fn = a.tc_f16 ? (const void*)deep_chain_tc_kernel<MODE, MCA_ACT_TANH, true>
                            : (const void*)deep_chain_tc_kernel<MODE, -1, false>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem);
  if (e != cudaSuccess) return e;
  DeepArgs args = a;
  void* params[] = {&args};
  return cudaLaunchKernel(fn, grid, dim3(kTcThreads), params, kTcSmem, s);
}

cudaError_t launch_deep_eval_tc(const DeepArgs& a, cudaStream_t s) {
  const int Kb = a.n_explicit > 0 ? a.n_explicit : a.Kb;
  return launch_tc<kChainEval>(a, dim3(Kb, a.ntiles), s);
}

cudaError_t launch_deep_commit_tc(const DeepArgs& a, cudaStream_t s) {
  return launch_tc<kChainCommit>(a, dim3(a.ntiles), s);
}

cudaError_t launch_deep_forward_tc(const DeepArgs& a, cudaStream_t s) {
  if (!a.tc_f16) return cudaErrorInvalidValue;
  const void* fn = (const void*)deep_chain_tc_kernel<kChainForward, MCA_ACT_TANH, true>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem);
  if (e != cudaSuccess) return e;
  DeepArgs args = a;
  void* params[] = {&args};
  return cudaLaunchKernel(fn, dim3(a.ntiles), dim3(kTcThreads), params, kTcSmem, s);
}

}  // namespace mca

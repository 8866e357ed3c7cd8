// Fields of a whole layer on the 5th-generation tensor cores: the forward pass over all samples
// (Section 2.1) that creation, mca_resync, mca_set_params and the channel trials run,
//   Z[M x Np] = W[M x K] act(B)[K x Np]       (feature-major fields, ld = Np; act = identity for X)
// as three tcgen05 MMAs per product: with W = W_hi + W_lo and A = act(B)^T = A_hi + A_lo,
// D = A_lo W_hi^T + A_hi W_lo^T + A_hi W_hi^T (the lo.lo term, ~2^-22 relative, dropped), accumulated in
// fp32 in tensor memory. The parts are fp16 or tf32, both 11 significant bits:
//  - fp16 costs half the MMAs and half the operand bytes, but has 5 exponent bits. Every sample's row of
//    A and every feature's row of W is scaled by a power of two that brings its largest magnitude to
//    [2^14, 2^15), taken back when the fields are written; then |x - hi - lo| <= 2^-22 |x| for values down
//    to 2^-17 of their row's largest, as with tf32, and 2^-39 of the largest below.
//  - tf32 for products too small to pay for finding the scales (kF16Macs), and where any row has
//    non-finite values, or more than wide_allowance of its non-zero values below 2^-17 of its largest: a field may
//    read only those. The scale kernels set a flag that the later kernels read.
//
// The operands are first written as split images in core-matrix order (mca_tc_layout.h; two fp16
// in the place of one tf32): A by blocks of 128 samples, W by blocks of 256 rows, both cut into K
// chunks of 32 (tf32: 16), each chunk the hi parts then the lo parts, so that one bulk copy moves one
// chunk. One CTA (4 warps) computes the transposed tile D^T[128 samples x 256 features]: thread 0 runs
// a two-stage ring of bulk copies (A chunk 16 KB + W chunk 32 KB per stage), warp 1 waits for each
// stage, issues its 6 MMAs (two K steps) and releases the stage through tcgen05.commit; after the last
// chunk every warp reads its 32 tensor-memory lanes (samples) and writes the fields, 32
// consecutive samples of one feature per store. 96 KB of shared memory and 256 tensor-memory columns
// per CTA, so two CTAs share an SM and one's epilogue overlaps the other's MMAs. CTAs run through the
// tiles in groups of kGGroup feature blocks, samples in the outer order, so that the CTAs at work share
// their operands in L2 (with samples innermost, A came from DRAM once per feature block).
//
// 784-16384 on 60000 samples: 2.7 ms (1.9 ms of it MMAs at 128 cycles each; the rest operands from L2
// and the epilogues that no other CTA hides), 5.1 ms with tf32 parts and samples innermost.
//
// Every wait is bounded (2 s); on a time-out the CTA records MCA_ERR_TIMEOUT, waits (bounded) for
// the copies it issued, frees its tensor memory and returns without writing.
#include <cuda_fp16.h>

#include "mca_device.cuh"
#include "mca_internal.h"
#include "mca_tc.cuh"
#include "mca_tc_layout.h"

namespace mca {

namespace {

constexpr int kGM = 128;                            // samples per tile (MMA M)
constexpr int kGN = 256;                            // features per tile (MMA N)
constexpr int kGK = 16;                             // K chunk of one stage: tf32, and twice that fp16
constexpr int kGGroup = 16;                         // feature blocks that CTAs take together
constexpr uint32_t kAHalf = kGM * kGK * 4;          // 8 KB: hi or lo of an A chunk
constexpr uint32_t kAChunk = 2 * kAHalf;
constexpr uint32_t kBHalf = kGN * kGK * 4;          // 16 KB: hi or lo of a W chunk
constexpr uint32_t kBChunk = 2 * kBHalf;
constexpr uint32_t kGStage = kAChunk + kBChunk;     // 48 KB
constexpr int kGStages = 2;
constexpr int kGThreads = 128;
constexpr int kGSmem = kGStages * kGStage;
// core-matrix strides (bytes): K-adjacent core matrices R * 16 apart, 8-row groups 128 apart
constexpr uint32_t kALBO = (kGM / 8) * 128, kASBO = 128;
constexpr uint32_t kBLBO = (kGN / 8) * 128, kBSBO = 128;
constexpr uint32_t kGIdesc16 = tc_idesc_f16(kGM, kGN), kGIdesc32 = tc_idesc_tf32(kGM, kGN);
// Multiply-adds from which fp16 parts pay for the scales, of the whole forward pass of 784-H-10 nets: 4000
// samples, H = 1024 (3.2e9) 91 us with tf32 parts, 90 us with fp16; 10000 samples (8e9) 160 and 147 us;
// 30000 samples, H = 2048 (4.8e10) 478 and 375 us; 4000 samples, H = 256 (8e8) 80 and 86 us.
constexpr double kF16Macs = 4294967296.0;

__device__ __forceinline__ void expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
               ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// Bulk copy whose bytes complete on `bar` (the arrival was counted by expect_tx).
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// Exponent e of the power of two that brings a row whose largest magnitude has these bits to
// [2^14, 2^15); 0 for infinities and NaN. Limited so that 2^e and the product of two scales' inverse
// halves are normal numbers.
__device__ __forceinline__ int row_exponent(unsigned int bits) {
  const int E = (int)(bits >> 23);
  return E == 255 ? 0 : min(14 + 127 - E, 126);
}
__device__ __forceinline__ float pow2(int e) { return __int_as_float((127 + e) << 23); }

// Of a row's values: how many are non-zero, and how many of these lie more than kWideGap binary orders
// below the largest (whose bits are top).
struct RowRange {
  unsigned int n, low;
  __device__ __forceinline__ void add(float v, unsigned int top) {
    const unsigned int m = __float_as_uint(fabsf(v));
    n += m != 0u;
    low += m != 0u && (m >> 23) + (unsigned int)kWideGap < (top >> 23);
  }
  __device__ __forceinline__ bool wide(unsigned int top) const {
    return top >> 23 == 255u || low > wide_allowance(n);
  }
};

// Eight consecutive k of row r (from k0, a multiple of 8) as 16-byte units: fp16 parts of the scaled
// values, or tf32 parts in two units each. Blocks of R rows, K columns.
__device__ __forceinline__ void store_split(const float (&v)[8], bool f16, float sc, int r, int k0,
                                            int R, int K, float* img) {
  if (f16) {
    union { __half h[8]; uint4 u; } hi, lo;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float x = v[q] * sc;
      hi.h[q] = __float2half_rn(x);
      lo.h[q] = __float2half_rn(x - __half2float(hi.h[q]));
    }
    const size_t o = tc_image_index(r, k0 >> 1, R, (K + 31) / 32 * 16);
    *reinterpret_cast<uint4*>(img + o) = hi.u;
    *reinterpret_cast<uint4*>(img + o + tc_image_lo(R)) = lo.u;
    return;
  }
  const int Kp = (K + kGK - 1) / kGK * kGK;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int k = k0 + 4 * u;
    if (k >= Kp) return;
    float hi[4], lo[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      hi[q] = tf32_rna(v[4 * u + q]);
      lo[q] = tf32_rna(v[4 * u + q] - hi[q]);
    }
    const size_t o = tc_image_index(r, k, R, Kp);
    *reinterpret_cast<float4*>(img + o) = make_float4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<float4*>(img + o + tc_image_lo(R)) = make_float4(lo[0], lo[1], lo[2], lo[3]);
  }
}

// The operands' form: tf32 without scales (wide null) or where a row's range is wide.
__device__ __forceinline__ bool use_f16(const int* wide) { return wide != nullptr && *wide == 0; }

__device__ __forceinline__ float act_value(const float* __restrict__ B, int k, int n, int Np, int act,
                                           float g) {
  const float v = B[(size_t)k * Np + n];
  return act >= 0 ? act_rt(act, v, g) : v;
}

// Scale exponents of the samples: 32 samples per CTA, 8 slices of k. (The second pass over a CTA's rows finds
// them in L2.)
__global__ void act_scale_kernel(const float* __restrict__ B, int K, int Np, int act, float g,
                                 int* __restrict__ ex, int* wide) {
  __shared__ unsigned int s_top[8][32];
  __shared__ RowRange s_r[8][32];
  const int lane = threadIdx.x & 31, p = threadIdx.x >> 5, n = blockIdx.x * 32 + lane;
  unsigned int top = 0u;
#pragma unroll 4
  for (int k = p; k < K; k += 8)
    top = max(top, __float_as_uint(fabsf(act_value(B, k, n, Np, act, g))));
  s_top[p][lane] = top;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 8; ++q) top = max(top, s_top[q][lane]);
  RowRange r{0u, 0u};
#pragma unroll 4
  for (int k = p; k < K; k += 8) r.add(act_value(B, k, n, Np, act, g), top);
  s_r[p][lane] = r;
  __syncthreads();
  if (p != 0) return;
#pragma unroll
  for (int q = 1; q < 8; ++q) {
    r.n += s_r[q][lane].n;
    r.low += s_r[q][lane].low;
  }
  ex[n] = row_exponent(top);
  if (r.wide(top)) *wide = 1;
}

// Scale exponents of W's rows: one warp per row.
__global__ void w_scale_kernel(const float* __restrict__ W, int M, int K, int* __restrict__ ex,
                               int* wide) {
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= M) return;
  unsigned int top = 0u;
#pragma unroll 4
  for (int k = lane; k < K; k += 32)
    top = max(top, __float_as_uint(fabsf(W[(size_t)row * K + k])));
  top = __reduce_max_sync(0xffffffffu, top);
  RowRange r{0u, 0u};
#pragma unroll 4
  for (int k = lane; k < K; k += 32) r.add(W[(size_t)row * K + k], top);
  r.n = __reduce_add_sync(0xffffffffu, r.n);
  r.low = __reduce_add_sync(0xffffffffu, r.low);
  if (lane == 0) {
    ex[row] = row_exponent(top);
    if (r.wide(top)) *wide = 1;
  }
}

// A image: act(B)^T split, blocks of 128 samples. Thread: one sample n, eight consecutive k.
__global__ void act_image_kernel(const float* __restrict__ B, int K, int Np, int act, float g,
                                 const int* __restrict__ ex, const int* wide,
                                 float* __restrict__ img) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  const int k0 = blockIdx.y * 8;
  if (n >= Np) return;
  const bool f16 = use_f16(wide);
  float v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q)
    v[q] = k0 + q < K ? act_value(B, k0 + q, n, Np, act, g) : 0.0f;
  store_split(v, f16, f16 ? pow2(ex[n]) : 1.0f, n, k0, kGM, K, img);
}

// W image: blocks of 256 rows. Thread: one row r, eight consecutive k.
__global__ void w_image_kernel(const float* __restrict__ W, int M, int K,
                               const int* __restrict__ ex, const int* wide,
                               float* __restrict__ img) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int k0 = blockIdx.y * 8;
  if (r >= M) return;
  const bool f16 = use_f16(wide);
  float v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = k0 + q < K ? W[(size_t)r * K + k0 + q] : 0.0f;
  store_split(v, f16, f16 ? pow2(ex[r]) : 1.0f, r, k0, kGN, K, img);
}

// The MMAs of one chunk (stage at sa / sb): lo hi, hi lo, hi hi for each of its two K steps.
template <bool F16>
__device__ __forceinline__ void chunk_mmas(uint32_t tmem, uint32_t sa, uint32_t sb, bool first) {
#pragma unroll
  for (int ks = 0; ks < 2; ++ks) {
    const uint64_t ahi = umma_desc(sa + (uint32_t)ks * 2u * kALBO, kALBO, kASBO);
    const uint64_t alo = umma_desc(sa + kAHalf + (uint32_t)ks * 2u * kALBO, kALBO, kASBO);
    const uint64_t bhi = umma_desc(sb + (uint32_t)ks * 2u * kBLBO, kBLBO, kBSBO);
    const uint64_t blo = umma_desc(sb + kBHalf + (uint32_t)ks * 2u * kBLBO, kBLBO, kBSBO);
    const uint32_t acc = first && ks == 0 ? 0u : 1u;
    if (F16) {
      mma_ss_f16(tmem, alo, bhi, kGIdesc16, acc);
      mma_ss_f16(tmem, ahi, blo, kGIdesc16, 1u);
      mma_ss_f16(tmem, ahi, bhi, kGIdesc16, 1u);
    } else {
      mma_ss(tmem, alo, bhi, kGIdesc32, acc);
      mma_ss(tmem, ahi, blo, kGIdesc32, 1u);
      mma_ss(tmem, ahi, bhi, kGIdesc32, 1u);
    }
  }
}

__global__ void __launch_bounds__(kGThreads) gemm_tc_kernel(const float* __restrict__ aimg,
                                                            const float* __restrict__ bimg,
                                                            const int* __restrict__ aex,
                                                            const int* __restrict__ bex,
                                                            const int* wide, int ns, int nf, int K,
                                                            float* __restrict__ Z, int ldz,
                                                            int* err) {
  extern __shared__ __align__(1024) unsigned char gsm[];
  __shared__ __align__(8) uint64_t s_full[kGStages], s_empty[kGStages], s_done;
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;
  __shared__ __align__(16) int s_bex[kGN];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = blockIdx.x / (ns * kGGroup), at = blockIdx.x - grp * ns * kGGroup;
  const int gn = min(kGGroup, nf - grp * kGGroup);
  const int bs = at / gn, bf = grp * kGGroup + at % gn;
  const bool f16 = use_f16(wide);
  const int nch = f16 ? (K + 2 * kGK - 1) / (2 * kGK) : (K + kGK - 1) / kGK;
  const unsigned char* ag =
      reinterpret_cast<const unsigned char*>(aimg) + (size_t)bs * nch * kAChunk;
  const unsigned char* bg =
      reinterpret_cast<const unsigned char*>(bimg) + (size_t)bf * nch * kBChunk;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;"
                 ::"r"(smem_u32(&s_tmem)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 32) {
    for (int q = 0; q < kGStages; ++q) {
      mbar_init(&s_full[q], 1);
      mbar_init(&s_empty[q], 1);
    }
    mbar_init(&s_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = 0;
  }
  for (int q = tid; q < kGN; q += kGThreads) s_bex[q] = f16 ? bex[bf * kGN + q] : 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const uint32_t sbase = smem_u32(gsm);

  if (tid == 0) {
    // producer: chunk c into stage c % 2 once the MMAs of chunk c - 2 released it
    int issued = 0;
    for (int c = 0; c < nch; ++c) {
      const int st = c % kGStages;
      if (c >= kGStages && !mbar_wait(&s_empty[st], (uint32_t)((c / kGStages) - 1) & 1u)) {
        s_fail = 1;
        break;
      }
      expect_tx(&s_full[st], kGStage);
      bulk_copy(sbase + (uint32_t)st * kGStage, ag + (size_t)c * kAChunk, kAChunk, &s_full[st]);
      bulk_copy(sbase + (uint32_t)st * kGStage + kAChunk, bg + (size_t)c * kBChunk, kBChunk,
                &s_full[st]);
      issued = c + 1;
    }
    // copies still in flight land before the CTA can leave (the consumer waits for the rest)
    for (int c = (issued > kGStages ? issued - kGStages : 0); c < issued; ++c)
      if (!mbar_wait(&s_full[c % kGStages], (uint32_t)(c / kGStages) & 1u)) s_fail = 1;
  } else if (warp == 1) {
    // MMA issuer
    for (int c = 0; c < nch; ++c) {
      const int st = c % kGStages;
      const bool ok = mbar_wait(&s_full[st], (uint32_t)(c / kGStages) & 1u);
      if (!__all_sync(0xffffffffu, ok)) {
        s_fail = 1;
        break;
      }
      tc_fence_after();
      const uint32_t sa = sbase + (uint32_t)st * kGStage, sb = sa + kAChunk;
      if (elect_one()) {
        if (f16)
          chunk_mmas<true>(tmem, sa, sb, c == 0);
        else
          chunk_mmas<false>(tmem, sa, sb, c == 0);
        umma_commit(&s_empty[st]);
      }
      __syncwarp();
    }
    if (elect_one()) umma_commit(&s_done);   // every MMA issued above has completed
  }
  __syncwarp();
  if (!mbar_wait(&s_done, 0u)) s_fail = 1;
  tc_fence_after();
  __syncthreads();
  if (!s_fail) {                           // the same value in every thread after the barrier
    const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
    const int n = bs * kGM + warp * 32 + lane;
    const int an = f16 ? aex[n] : 0;
    float* zc = Z + (size_t)bf * kGN * ldz + n;
    for (int c0 = 0; c0 < kGN; c0 += 16) {
      float v[16];
      tmem_ld16(tmem + lane_base + (uint32_t)c0, v);
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int e = -(an + s_bex[c0 + q]), h = e >> 1;   // two factors: neither leaves the range
        zc[(size_t)(c0 + q) * ldz] = v[q] * pow2(h) * pow2(e - h);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem));
  if (tid == 0 && s_fail) atomicCAS(err, 0, (int)MCA_ERR_TIMEOUT);
}

}  // namespace

bool gemm_tc_ok(int M, int K, int Np) { return M > 0 && M % kGN == 0 && K >= 1 && Np % kGM == 0; }

size_t gemm_tc_image_bytes(int M, int K, int Np) {
  const size_t nch = (size_t)(K + kGK - 1) / kGK;
  return nch * ((size_t)(Np / kGM) * kAChunk + (size_t)(M / kGN) * kBChunk) +
         sizeof(int) * ((size_t)Np + (size_t)M + 1);
}

cudaError_t launch_gemm_tc(const float* W, int M, int K, const float* B, int act, float g,
                           float* Z, int Np, float* img, int* err, cudaStream_t s) {
  if (!gemm_tc_ok(M, K, Np)) return cudaErrorInvalidValue;
  const int nch = (K + kGK - 1) / kGK, ns = Np / kGM, nf = M / kGN;
  float* aimg = img;
  float* bimg = aimg + (size_t)nch * (size_t)ns * (kAChunk / 4);
  int* aex = reinterpret_cast<int*>(bimg + (size_t)nch * (size_t)nf * (kBChunk / 4));
  int* bex = aex + Np;
  int* wide = nullptr;
  cudaError_t e;
  if ((double)M * (double)Np * (double)K >= kF16Macs) {
    wide = bex + M;
    e = cudaMemsetAsync(wide, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    act_scale_kernel<<<Np / 32, 256, 0, s>>>(B, K, Np, act, g, aex, wide);
    w_scale_kernel<<<(M + 7) / 8, 256, 0, s>>>(W, M, K, bex, wide);
  }
  const int units = wide ? (K + 31) / 32 * 4 : nch * 2;   // of eight k, padding included
  act_image_kernel<<<dim3((Np + 127) / 128, units), 128, 0, s>>>(
      B, K, Np, act, g, aex, wide, aimg);
  w_image_kernel<<<dim3((M + 127) / 128, units), 128, 0, s>>>(
      W, M, K, bex, wide, bimg);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(gemm_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGSmem);
  if (e != cudaSuccess) return e;
  gemm_tc_kernel<<<(unsigned int)ns * (unsigned int)nf, kGThreads, kGSmem, s>>>(
      aimg, bimg, aex, bex, wide, ns, nf, K, Z, Np, err);
  return cudaGetLastError();
}

}  // namespace mca

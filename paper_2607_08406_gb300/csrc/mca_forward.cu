// Full forward pass of the single-hidden-layer net and the creation-time data preparation:
// X -> feature-major XT, the CSR of X by input feature (plus per-range offsets and sector counts),
// parameter initialisation, z1 = W1 X^T (SIMT SGEMM), output fields, per-sample losses and S.
#include <algorithm>
#include <cstdio>

#include <cooperative_groups.h>

#include "mca_device.cuh"
#include "mca_internal.h"

namespace mca {

// ------------------------------------------------------------------------------------------------
// Full forward pass (resync): z1 = W1 X^T (SGEMM), then output fields, losses and S.
// ------------------------------------------------------------------------------------------------

// XT[i, n] = X[n, i] for n < N, 0 in the padding columns.
__global__ void transpose_pad_kernel(const float* __restrict__ X, int N, int D,
                                     float* __restrict__ XT, int Np) {
  __shared__ float tile[32][33];
  const int n0 = blockIdx.x * 32, i0 = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int n = n0 + r, i = i0 + threadIdx.x;
    tile[r][threadIdx.x] = (n < N && i < D) ? X[(size_t)n * D + i] : 0.0f;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int i = i0 + r, n = n0 + threadIdx.x;
    if (i < D && n < Np) XT[(size_t)i * Np + n] = tile[threadIdx.x][r];
  }
}

__global__ void csr_count_kernel(const float* __restrict__ XT, int Np, int N, int* cnt) {
  const float* row = XT + (size_t)blockIdx.x * Np;
  int c = 0;
  for (int n0 = 0; n0 < N; n0 += blockDim.x) {
    const int n = n0 + threadIdx.x;
    c += __syncthreads_count(n < N && row[n] != 0.0f);
  }
  if (threadIdx.x == 0) cnt[blockIdx.x] = c;
}

// One CTA per feature; block-wide compaction keeps entries in ascending sample order.
__global__ void csr_fill_kernel(const float* __restrict__ XT, int Np, int N, const int* off,
                                int* xs_n, float* xs_v) {
  __shared__ int wcount[32];
  __shared__ int s_base;
  const float* row = XT + (size_t)blockIdx.x * Np;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (threadIdx.x == 0) s_base = off[blockIdx.x];
  __syncthreads();
  for (int n0 = 0; n0 < N; n0 += blockDim.x) {
    const int n = n0 + threadIdx.x;
    const float v = n < N ? row[n] : 0.0f;
    const bool nz = v != 0.0f;
    const unsigned int m = __ballot_sync(0xffffffffu, nz);
    if (lane == 0) wcount[warp] = __popc(m);
    __syncthreads();
    int before = 0, tot = 0;
    for (int w = 0; w < nw; ++w) {
      if (w < warp) before += wcount[w];
      tot += wcount[w];
    }
    const int pos = s_base + before + __popc(m & ((1u << lane) - 1u));
    if (nz) {
      xs_n[pos] = n;
      xs_v[pos] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0) s_base += tot;
    __syncthreads();
  }
}

// Distinct 32-byte sectors (8 samples) of a z1 row holding feature i's entries.
__global__ void csr_sectors_kernel(const int* __restrict__ off, const int* __restrict__ xs_n,
                                   int* sect) {
  const int s = off[blockIdx.x], e = off[blockIdx.x + 1];
  int c = 0;
  for (int p0 = s; p0 < e; p0 += blockDim.x) {
    const int p = p0 + threadIdx.x;
    c += __syncthreads_count(p < e && (p == s || (xs_n[p] >> 3) != (xs_n[p - 1] >> 3)));
  }
  if (threadIdx.x == 0) sect[blockIdx.x] = c;
}

// roff[i * (NR + 1) + r] = first entry of feature i whose sample is >= r * RS (binary search over
// the feature's ascending sample list); roff[i * (NR + 1) + NR] = end of the feature's entries.
__global__ void csr_range_offsets_kernel(const int* __restrict__ off, const int* __restrict__ xs_n,
                                         int NR, int RS, int* roff) {
  const int i = blockIdx.x;
  const int b = off[i], e = off[i + 1];
  for (int r = threadIdx.x; r <= NR; r += blockDim.x) {
    int lo = b, hi = e;
    if (r < NR) {
      const long long s = (long long)r * RS;
      while (lo < hi) {
        const int mid = lo + ((hi - lo) >> 1);
        if (xs_n[mid] < s)
          lo = mid + 1;
        else
          hi = mid;
      }
    } else {
      lo = e;
    }
    roff[(size_t)i * (NR + 1) + r] = lo;
  }
}

__global__ void count_nonfinite_kernel(const float* __restrict__ p, size_t n, int* out) {
  int bad = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    bad |= !isfinite(p[i]);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(out, 1);
}

__global__ void abs_max_kernel(const float* __restrict__ p, size_t n, int* out) {
  int m = 0;                         // the bits of non-negative floats order like the floats
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    m = max(m, __float_as_int(fabsf(p[i])));
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

__global__ void init_layer_kernel(int wkind, float scale, const float* __restrict__ src,
                                  const signed char* __restrict__ mask, size_t n, float* w_eff,
                                  signed char* code, float* wfix) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const float v = src[i];
    if (wkind == MCA_W_TERNARY_I8) {
      const int t = (int)v;
      code[i] = (signed char)t;
      w_eff[i] = __fmul_rn(scale, (float)t);
    } else if (wkind == MCA_W_MASKED_FP32) {
      const int m = mask ? (mask[i] != 0) : 1;
      wfix[i] = v;
      code[i] = (signed char)m;
      w_eff[i] = m ? v : 0.0f;
    } else {
      w_eff[i] = v;
    }
  }
}

// C[M x Ncol] = A[M x K] * B[K x Ncol], row-major, fp32 FMA in ascending k. Ncol % 128 == 0,
// ldb and ldc multiples of 4. ACTB: the B operand enters as act(B) (the previous layer's activations
// from its fields).
//
// 256 threads compute a tile of 16 R x 16 R outputs, R x R per thread. The next 16 k are in flight (in
// registers) while a chunk is multiplied out of one of two buffers, one barrier per chunk; products come
// in pairs of columns, each rounded as a single one. Small products are bounded by latency, so the
// tile is the largest one whose CTAs fill the GPU (sgemm_tile). The forward pass of 784-64-10 on 1000
// samples takes 65 us (152 us with tiles of 128 throughout, one chunk of 8 k at a time), of 784-100x5-10
// on 3001 samples 125 us (258 us), of 391-1001-7 on 12347 samples 285 us (336 us).
constexpr int kSgK = 16;

// Row or column of value q of thread t (of 16): groups of four for the vector loads.
template <int R>
__device__ __forceinline__ int sg_at(int t, int q) {
  return R == 8 ? (q >> 2) * 64 + t * 4 + (q & 3) : t * R + q;
}

template <int R>
__device__ __forceinline__ void sg_load(const float* p, int t, float (&v)[R]) {
  if constexpr (R == 2) {
    const float2 x = *reinterpret_cast<const float2*>(p + 2 * t);
    v[0] = x.x;
    v[1] = x.y;
  } else {
#pragma unroll
    for (int g = 0; g < R / 4; ++g) {
      const float4 x = *reinterpret_cast<const float4*>(p + 64 * g + 4 * t);
      v[4 * g] = x.x;
      v[4 * g + 1] = x.y;
      v[4 * g + 2] = x.z;
      v[4 * g + 3] = x.w;
    }
  }
}

template <int R, bool ACTB>
__global__ void __launch_bounds__(256, R == 8 ? 2 : 4) sgemm_nn_kernel(
    int M, int K, const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb,
    float* __restrict__ C, int ldc, int bact, float bg) {
  constexpr int BM = 16 * R, BN = 16 * R;
  constexpr int NB = (kSgK * BN / 4 + 255) / 256;   // 16-byte units of B per thread
  __shared__ __align__(16) float As[2][kSgK][BM + 4];
  __shared__ __align__(16) float Bs[2][kSgK][BN];
  const int tid = threadIdx.x;
  const int bm = blockIdx.y * BM, bn = blockIdx.x * BN;
  const int tr = tid / 16, tc = tid % 16;
  float2 acc[R][R / 2];
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < R / 2; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
  float an[R];                                      // k = tid % 16 of rows tid / 16 + 16 u
  float4 bv[NB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const int m = bm + tr + 16 * u, kk = k0 + tc;
      an[u] = m < M && kk < K ? A[(size_t)m * lda + kk] : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int e = tid + 256 * u, kk = k0 + e / (BN / 4), col = e % (BN / 4) * 4;
      bv[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (e < kSgK * BN / 4 && kk < K)
        bv[u] = *reinterpret_cast<const float4*>(B + (size_t)kk * ldb + bn + col);
    }
  };
  fetch(0);
  int buf = 0;
#pragma unroll 1
  for (int k0 = 0; k0 < K; k0 += kSgK) {
#pragma unroll
    for (int u = 0; u < R; ++u) As[buf][tc][tr + 16 * u] = an[u];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int e = tid + 256 * u, kk = e / (BN / 4), col = e % (BN / 4) * 4;
      if (e >= kSgK * BN / 4) continue;
      float4 v = bv[u];
      if (ACTB && k0 + kk < K) {
        v.x = act_rt(bact, v.x, bg);
        v.y = act_rt(bact, v.y, bg);
        v.z = act_rt(bact, v.z, bg);
        v.w = act_rt(bact, v.w, bg);
      }
      *reinterpret_cast<float4*>(&Bs[buf][kk][col]) = v;
    }
    __syncthreads();
    if (k0 + kSgK < K) fetch(k0 + kSgK);
#pragma unroll
    for (int kk = 0; kk < kSgK; ++kk) {
      float ra[R], rb[R];
      sg_load<R>(As[buf][kk], tr, ra);
      sg_load<R>(Bs[buf][kk], tc, rb);
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R / 2; ++j)
          acc[i][j] = fma2(make_float2(ra[i], ra[i]), make_float2(rb[2 * j], rb[2 * j + 1]),
                           acc[i][j]);
    }
    buf ^= 1;
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int m = bm + sg_at<R>(tr, i);
    if (m >= M) continue;
    float* crow = C + (size_t)m * ldc + bn;
#pragma unroll
    for (int j = 0; j < R / 2; ++j)
      *reinterpret_cast<float2*>(crow + sg_at<R>(tc, 2 * j)) = acc[i][j];
  }
}

// Output fields z2[:, n] = W2 f(z1[:, n]), the sample's loss, and its label. One CTA per 32 samples
// (lane = sample), its 16 warps taking 32-row chunks of z1 in turn; the warps' partial sums are added
// in warp order. Reading z1 once bounds it (3.9 GB for 16384 hidden neurons and 60000 samples: 0.58 ms
// at the copy bandwidth). One thread per sample walking every hidden neuron left 469 CTAs of 4 warps
// waiting for one load at a time (5.28 ms); splitting the neurons over the warps, with 16 rows in
// flight per warp, takes 1.11 ms.
constexpr int kOutWarps = 16, kOutRows = 32;

template <int ACT1, int NC>
__global__ void __launch_bounds__(kOutWarps * 32, 2) mlp2_outputs_kernel(
    Mlp2Args a, const int* __restrict__ y) {
  constexpr int M = NC > 0 ? NC : kMaxC;
  const int C = NC > 0 ? NC : a.C;
  __shared__ __align__(16) float s_w[kOutWarps][M][kOutRows];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = blockIdx.x * 32 + lane;              // < Np: always in the arrays
  const float* z = a.z1 + n;
  float acc[M];
#pragma unroll
  for (int k = 0; k < M; ++k) acc[k] = 0.0f;
  for (int j0 = warp * kOutRows; j0 < a.H; j0 += kOutWarps * kOutRows) {
    __syncwarp();
#pragma unroll
    for (int k = 0; k < M; ++k)
      if (k < C) s_w[warp][k][lane] = j0 + lane < a.H ? a.w2[(size_t)k * a.H + j0 + lane] : 0.0f;
    __syncwarp();
#pragma unroll 1
    for (int h = 0; h < kOutRows; h += 16) {
      float v[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) v[q] = z[(size_t)min(j0 + h + q, a.H - 1) * a.Np];
#pragma unroll
      for (int q = 0; q < 16; ++q)                   // (rows past the last: 0 times infinity is not 0)
        v[q] = j0 + h + q < a.H ? act<ACT1>(v[q], a.g1, a.act1) : 0.0f;
#pragma unroll
      for (int k = 0; k < M; ++k) {
        if (k < C) {
#pragma unroll
          for (int q = 0; q < 16; q += 4) {
            const float4 w = *reinterpret_cast<const float4*>(&s_w[warp][k][h + q]);
            acc[k] = fmaf(w.x, v[q], acc[k]);
            acc[k] = fmaf(w.y, v[q + 1], acc[k]);
            acc[k] = fmaf(w.z, v[q + 2], acc[k]);
            acc[k] = fmaf(w.w, v[q + 3], acc[k]);
          }
        }
      }
    }
  }
  __syncwarp();
#pragma unroll
  for (int k = 0; k < M; ++k) s_w[warp][k][lane] = acc[k];
  __syncthreads();
  if (warp == 0 && n < a.N) {
    float zz[kMaxC];
#pragma unroll
    for (int k = 0; k < kMaxC; ++k) {
      zz[k] = 0.0f;
      if (k < M && k < C) {
#pragma unroll
        for (int w = 0; w < kOutWarps; ++w) zz[k] += s_w[w][k < M ? k : 0][lane];
      }
    }
    const int yn = y[n];
    const float ln = sample_loss<-1, -1, kMaxC, true>(zz, C, yn, a.g2, a.act2, a.loss);
    store_srec(a.srec, a.Np, n, zz, ln, yn);
  }
}

// S = sum_n loss_n in fp64, fixed order: a cluster of 8 CTAs, CTA r summing the r-th eighth and CTA 0
// adding the eight partial sums. The fp64 additions bound it (one SM has few fp64 lanes): 33 us with
// one CTA at 60000 samples, 11 us with eight.
constexpr int kSumCtas = 8;

__global__ void __cluster_dims__(kSumCtas, 1, 1) __launch_bounds__(1024)
    sum_loss_kernel(const float* __restrict__ ell, int N, DevState* st) {
  namespace cg = cooperative_groups;
  __shared__ double red[32];
  __shared__ double part;
  cg::cluster_group cl = cg::this_cluster();
  const int per = (N + kSumCtas - 1) / kSumCtas;
  const int b = min(N, (int)blockIdx.x * per), e = min(N, b + per);
  double s = 0.0;
#pragma unroll 4
  for (int n = b + threadIdx.x; n < e; n += blockDim.x) s += (double)ell[n];
  s = block_sum_d(s, red);
  if (threadIdx.x == 0) part = s;
  cl.sync();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < kSumCtas; ++q) t += *cl.map_shared_rank(&part, q);
    st->S = t;
  }
  cl.sync();                                         // the partial sums outlive their readers
}

// ------------------------------------------------------------------------------------------------
// Launchers
// ------------------------------------------------------------------------------------------------
cudaError_t launch_transpose_pad(const float* X, int N, int D, float* XT, int Np, cudaStream_t s) {
  dim3 grid((Np + 31) / 32, (D + 31) / 32), block(32, 8);
  transpose_pad_kernel<<<grid, block, 0, s>>>(X, N, D, XT, Np);
  return cudaGetLastError();
}

cudaError_t launch_csr_count(const float* XT, int Np, int N, int D, int* cnt, cudaStream_t s) {
  csr_count_kernel<<<D, 256, 0, s>>>(XT, Np, N, cnt);
  return cudaGetLastError();
}

cudaError_t launch_csr_fill(const float* XT, int Np, int N, int D, const int* off, int* xs_n,
                            float* xs_v, cudaStream_t s) {
  csr_fill_kernel<<<D, 1024, 0, s>>>(XT, Np, N, off, xs_n, xs_v);
  return cudaGetLastError();
}

cudaError_t launch_csr_sectors(const int* off, const int* xs_n, int D, int* sect, cudaStream_t s) {
  csr_sectors_kernel<<<D, 256, 0, s>>>(off, xs_n, sect);
  return cudaGetLastError();
}

cudaError_t launch_csr_range_offsets(const int* off, const int* xs_n, int D, int NR, int RS,
                                     int* roff, cudaStream_t s) {
  csr_range_offsets_kernel<<<D, 256, 0, s>>>(off, xs_n, NR, RS, roff);
  return cudaGetLastError();
}

cudaError_t launch_count_nonfinite(const float* p, size_t n, int* out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int grid = (int)std::min<size_t>(4096, (n + 255) / 256);
  count_nonfinite_kernel<<<grid, 256, 0, s>>>(p, n, out);
  return cudaGetLastError();
}

cudaError_t launch_abs_max(const float* p, size_t n, int* out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int grid = (int)std::min<size_t>(1024, (n + 255) / 256);
  abs_max_kernel<<<grid, 256, 0, s>>>(p, n, out);
  return cudaGetLastError();
}

cudaError_t launch_init_layer(int wkind, float scale, const float* src, const signed char* mask,
                              size_t n, float* w_eff, signed char* code, float* wfix,
                              cudaStream_t s) {
  const int grid = (int)std::min<size_t>(4096, (n + 255) / 256);
  init_layer_kernel<<<grid, 256, 0, s>>>(wkind, scale, src, mask, n, w_eff, code, wfix);
  return cudaGetLastError();
}

// R of the SGEMM's tiles: 8 while two CTAs per SM have one, then 4 while every SM does, else 2.
static int sgemm_tile(int M, int Ncol) {
  auto ctas = [&](int t) { return (long long)(Ncol / t) * ((M + t - 1) / t); };
  return ctas(128) >= 304 ? 8 : ctas(64) >= 152 ? 4 : 2;
}

template <bool ACTB>
static cudaError_t launch_sgemm(int M, int Ncol, int K, const float* A, int lda, const float* B,
                                int ldb, float* C, int ldc, int bact, float bg, cudaStream_t s) {
  const int R = sgemm_tile(M, Ncol), t = 16 * R;
  const dim3 grid(Ncol / t, (M + t - 1) / t);
  auto fn = R == 8 ? sgemm_nn_kernel<8, ACTB>
            : R == 4 ? sgemm_nn_kernel<4, ACTB> : sgemm_nn_kernel<2, ACTB>;
  fn<<<grid, 256, 0, s>>>(M, K, A, lda, B, ldb, C, ldc, bact, bg);
  return cudaGetLastError();
}

cudaError_t launch_sgemm_nn(int M, int Ncol, int K, const float* A, int lda, const float* B,
                            int ldb, float* C, int ldc, cudaStream_t s) {
  return launch_sgemm<false>(M, Ncol, K, A, lda, B, ldb, C, ldc, 0, 0.0f, s);
}

// Fields of deep layer l from the previous layer (or X for l = 0): Z_l = W_l act_{l-1}(Z_{l-1}).
cudaError_t launch_deep_forward_layer(const DeepArgs& a, int l, cudaStream_t s) {
  const int M = a.n_out[l], K = a.n_in[l];
  if (l == 0) return launch_sgemm_nn(M, a.Np, K, a.w[0], K, a.XT, a.Np, a.Z[0], a.Np, s);
  return launch_sgemm<true>(M, a.Np, K, a.w[l], K, a.Z[l - 1], a.Np, a.Z[l], a.Np, a.act[l - 1],
                            a.g[l - 1], s);
}

cudaError_t launch_sum_loss(const float* ell, int N, DevState* st, cudaStream_t s) {
  sum_loss_kernel<<<kSumCtas, 1024, 0, s>>>(ell, N, st);
  return cudaGetLastError();
}

// Output-field kernel variants: the hidden transfer functions and class count of the trial loop's.
using OutFn = void (*)(Mlp2Args, const int*);

template <int NC>
static OutFn pick_outputs(int act1) {
  switch (act1) {
    case MCA_ACT_TANH: return mlp2_outputs_kernel<MCA_ACT_TANH, NC>;
    case MCA_ACT_GAUSSIAN: return mlp2_outputs_kernel<MCA_ACT_GAUSSIAN, NC>;
    case MCA_ACT_RELU: return mlp2_outputs_kernel<MCA_ACT_RELU, NC>;
    default: return mlp2_outputs_kernel<-1, NC>;
  }
}

cudaError_t launch_mlp2_outputs(const Mlp2Args& a, const int* y, cudaStream_t s) {
  const OutFn fn = a.C == 10 ? pick_outputs<10>(a.act1) : pick_outputs<-1>(a.act1);
  fn<<<(a.N + 31) / 32, kOutWarps * 32, 0, s>>>(a, y);
  return cudaGetLastError();
}

}  // namespace mca

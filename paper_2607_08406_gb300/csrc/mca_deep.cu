// Deep MLP path of the MCA trial loop (three or more weight layers; the 24 x 256 tanh net).
//
// Cached state: the fields Z_l = W_l a_{l-1} of every layer for all samples ([n_out x Np],
// feature-major) and every sample's loss. A candidate W_l[j, i] -> W_l[j, i] + delta changes
//   row j of layer l:      z'_l[j, n]  = z_l[j, n] + delta a_{l-1}[i, n]            (Section 2.4)
//   layer l+1 (rank-1):    Z'_{l+1}    = Z_{l+1} + W_{l+1}[:, j] (f(z'_l[j]) - f(z_l[j]))
//   layers m >= l+2:       Z'_m        = Z_m + W_m (f(Z'_{m-1}) - f(Z_{m-1}))
// i.e. the dense recomputation from l+2 on is carried as a change: a sample whose activations did not
// change contributes exactly zero, and the commit writes exactly what the evaluation computed.
//
// Per batch the host launches three kernels:
//   deep_eval     grid (K, tiles): CTA (k, t) runs candidate k's chain over tile t's samples (32 or 64),
//                 the change matrix staying in shared memory from layer to layer, and writes one
//                 partial loss change per (candidate, tile) -- a fixed computation, independent of K
//   deep_decide   one CTA: fixed-order (compensated fp32) sums, lowest-index candidate with
//                 dS <= theta (Eq. 6: theta = 0; Eq. 7: the trial's Metropolis threshold), trace,
//                 statistics, weight update
//   deep_commit   grid (tiles): the accepted candidate's chain with writes
#include <algorithm>
#include <cstdio>

#include "mca_deep.cuh"
#include "mca_device.cuh"
#include "mca_internal.h"

namespace mca {

// Transfer function of a hidden layer: tanh in place, any other called.
__device__ __forceinline__ float hidden_act(int act, float z, float g) {
  return act == MCA_ACT_TANH ? tanh_exp(z) : act_call(act, z, g);
}

// Chunk of kDeepKC weights W[row][k0 ..] of one row into registers (0 past the last column).
__device__ __forceinline__ void load_row_chunk(const float* W, int row, int K, int k0,
                                               float (&w)[kDeepKC]) {
  const float* src = W + (size_t)row * K + k0;
  if (k0 + kDeepKC <= K && (K & 3) == 0) {
#pragma unroll
    for (int v = 0; v < kDeepKC / 4; ++v) {
      const float4 w4 = *reinterpret_cast<const float4*>(src + 4 * v);
      w[4 * v] = w4.x;
      w[4 * v + 1] = w4.y;
      w[4 * v + 2] = w4.z;
      w[4 * v + 3] = w4.w;
    }
  } else {
#pragma unroll
    for (int v = 0; v < kDeepKC; ++v) w[v] = k0 + v < K ? src[v] : 0.0f;
  }
}

// Commit of an accepted candidate whose evaluation kept its fields: samples n0 .. n0 + TS of its scratch
// slot (row j of its layer, every row of the later layers, the losses) to the cached state. (Running the
// chain again took as long as the evaluation: decision and commit of a 784-100x5-10 batch on 3001 samples
// 35 us, with the copy 24 us.)
template <int TS>
__device__ void adopt_tile(const DeepArgs& a, const DeepCand& c, float* const* sk, int n0) {
  const int t = threadIdx.x % TS, p = threadIdx.x / TS, n = n0 + t;
  constexpr int PARTS = kDeepThreads / TS;
  if (n >= a.N) return;
  const size_t Np = (size_t)a.Np;
  if (p == 0) {
    a.Z[c.layer][(size_t)c.row * Np + n] = sk[c.layer][(size_t)c.row * Np + n];
    a.ell[n] = sk[a.L][n];
  }
  for (int m = c.layer + 1; m < a.L; ++m) {
    const float* src = sk[m] + n;
    float* dst = a.Z[m] + n;
    const int M = a.n_out[m];
#pragma unroll 8
    for (int r = p; r < M; r += PARTS) dst[r * Np] = src[r * Np];
  }
}

// One CTA per (candidate, tile of 16 S samples): thread (ty, tx) computes R rows x S samples of a dense
// layer, so that 16 R >= the widest layer. What bounds a chain is the latency of its layers, one after
// another: the next weight chunk is in flight (in registers) while one is multiplied, a layer's
// cached fields are loaded before its product, and small nets (fewer than one 64-sample tile per SM)
// use tiles of 32. (With 256 rows and 64 samples whatever the widths, no load ahead of its use and
// one thread per sample in the output layer, five layers of 100 on 3001 samples took 156 us per batch;
// now 74 us.)
template <bool COMMIT, int R, int S>
__global__ void __launch_bounds__(kDeepThreads) deep_chain_kernel(DeepArgs a) {
  constexpr int TS = 16 * S, ROWS = 16 * R;
  extern __shared__ __align__(16) float sm[];
  float* Ds = sm;                                   // [kDeepMaxWidth][TS] activation changes
  float* Ws = sm + kDeepMaxWidth * TS;              // two weight chunks [kDeepKC][ROWS]
  __shared__ DeepCand s_cand;
  __shared__ float s_da[TS];
  __shared__ float s_red[32];
  const int tid = threadIdx.x;
  const int k = COMMIT ? 0 : blockIdx.x;
  const int tile = COMMIT ? blockIdx.x : blockIdx.y;
  const int n0 = tile * TS;
  if (COMMIT && a.ctl->kstar < 0) return;
  if (tid == 0) s_cand = COMMIT ? a.ctl->acc : deep_candidate(a, k);
  __syncthreads();
  const DeepCand c = s_cand;
  float* part = a.partial + (size_t)k * a.ntiles + tile;
  if (!c.valid || c.delta == 0.0f) {
    if (!COMMIT && tid == 0) *part = 0.0f;
    return;
  }
  const int L = a.L, l = c.layer, j = c.row, i = c.col;
  const int Np = a.Np, N = a.N;
  float dl = 0.0f;
  if (COMMIT && a.ctl->kstar < a.nscr) {
    adopt_tile<TS>(a, c, a.scr + (size_t)a.ctl->kstar * (L + 1), n0);
    return;
  }
  // the candidate's scratch slot (pointers per layer, then the losses), if it has one
  float* const* sk = !COMMIT && k < a.nscr ? a.scr + (size_t)k * (L + 1) : nullptr;
  float* const sk_z = sk ? sk[L - 1] : nullptr;
  float* const sk_l = sk ? sk[L] : nullptr;

  // ---- row j of layer l
  if (tid < TS) {
    const int n = n0 + tid;
    float da = 0.0f;
    if (n < N) {
      const float v = l == 0 ? a.XT[(size_t)i * Np + n]
                             : hidden_act(a.act[l - 1], a.Z[l - 1][(size_t)i * Np + n], a.g[l - 1]);
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
        dl = out_delta<COMMIT>(a, n, zz, zn != z, sk_z, sk_l);
      } else {
        da = hidden_act(a.act[l], zn, a.g[l]) - hidden_act(a.act[l], z, a.g[l]);
        if (COMMIT) *zp = zn;
        if (sk) sk[l][(size_t)j * Np + n] = zn;
      }
    }
    s_da[tid] = da;
  }
  __syncthreads();

  if (l < L - 1) {
    // ---- layer l+1: rank-1 change through column j of W_{l+1}
    const int m1 = l + 1;
    const float* W1 = a.w[m1];
    const int K1 = a.n_in[m1];
    if (m1 == L - 1) {
      if (tid < TS) {
        const int n = n0 + tid;
        const float da = s_da[tid];
        if (n < N && (da != 0.0f || sk)) {
          float zz[kMaxC];
          bool changed = false;
#pragma unroll
          for (int q = 0; q < kMaxC; ++q) {
            if (q < a.C) {
              const float zo = a.Z[m1][(size_t)q * Np + n];
              zz[q] = da != 0.0f ? fmaf(W1[(size_t)q * K1 + j], da, zo) : zo;
              changed |= zz[q] != zo;
            } else {
              zz[q] = 0.0f;
            }
          }
          dl = out_delta<COMMIT>(a, n, zz, changed, sk_z, sk_l);
        }
      }
    } else {
      const int M = a.n_out[m1], act1 = a.act[m1];
      const float g1 = a.g[m1];
      float* Z1 = a.Z[m1];
      float* const S1 = sk ? sk[m1] : nullptr;
#pragma unroll 1
      for (int e0 = tid; e0 < M * TS; e0 += 4 * kDeepThreads) {
        float zo[4], w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {               // n < Np: always in the arrays
          const int e = e0 + u * kDeepThreads, r = min(e / TS, M - 1);
          zo[u] = Z1[(size_t)r * Np + n0 + e % TS];
          w[u] = W1[(size_t)r * K1 + j];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int e = e0 + u * kDeepThreads, r = e / TS, t = e % TS, n = n0 + t;
          if (e >= M * TS) break;
          const float da = s_da[t];
          float d = 0.0f, zn = zo[u];
          if (n < N && da != 0.0f) {
            zn = fmaf(w[u], da, zo[u]);
            if (COMMIT) Z1[(size_t)r * Np + n] = zn;
            d = hidden_act(act1, zn, g1) - hidden_act(act1, zo[u], g1);
          }
          if (S1 && n < N) S1[(size_t)r * Np + n] = zn;
          Ds[e] = d;
        }
      }
      __syncthreads();

      // ---- layers l+2 .. L-2: Z'_m = Z_m + W_m D, D <- f(Z'_m) - f(Z_m)
      const int ty = tid >> 4, tx = tid & 15;
      const int wrow = tid < ROWS ? tid : 0;         // the row whose weights this thread stages
      for (int m = l + 2; m < L - 1; ++m) {
        const float* Wm = a.w[m];
        const int Mm = a.n_out[m], Km = a.n_in[m];
        float* Zm = a.Z[m];
        float* const Sm = sk ? sk[m] : nullptr;
        constexpr bool kAhead = R * S <= 32;         // registers for the cached fields meanwhile
        float zf[kAhead ? R : 1][S];
        if (kAhead) {
#pragma unroll
          for (int q = 0; q < R; ++q)
#pragma unroll
            for (int cc = 0; cc < S; ++cc)
              zf[kAhead ? q : 0][cc] =
                  Zm[(size_t)min(ty * R + q, Mm - 1) * Np + n0 + tx * S + cc];
        }
        float acc[R][S];
#pragma unroll
        for (int q = 0; q < R; ++q)
#pragma unroll
          for (int cc = 0; cc < S; ++cc) acc[q][cc] = 0.0f;
        float wn[kDeepKC];
        const bool stage = tid < Mm;                 // Mm <= ROWS
        if (stage) load_row_chunk(Wm, wrow, Km, 0, wn);
        int buf = 0;
#pragma unroll 1
        for (int k0 = 0; k0 < Km; k0 += kDeepKC) {
          const int kn = min(kDeepKC, Km - k0);
          float* Wb = Ws + buf * kDeepKC * ROWS;
          if (stage) {
#pragma unroll
            for (int v = 0; v < kDeepKC; ++v) Wb[v * ROWS + tid] = wn[v];
          }
          __syncthreads();
          if (stage && k0 + kDeepKC < Km) load_row_chunk(Wm, wrow, Km, k0 + kDeepKC, wn);
          if (ty * R < Mm) {
#pragma unroll 4
            for (int kk = 0; kk < kn; ++kk) {
              float b[S], av[R];
              const float* dr = &Ds[(k0 + kk) * TS + tx * S];
              if constexpr (S == 4) {
                const float4 v = *reinterpret_cast<const float4*>(dr);
                b[0] = v.x;
                b[1] = v.y;
                b[2] = v.z;
                b[3] = v.w;
              } else {
                const float2 v = *reinterpret_cast<const float2*>(dr);
                b[0] = v.x;
                b[1] = v.y;
              }
              const float* wr = &Wb[kk * ROWS + ty * R];
#pragma unroll
              for (int v4 = 0; v4 < R / 4; ++v4) {
                const float4 w4 = *reinterpret_cast<const float4*>(wr + 4 * v4);
                av[4 * v4] = w4.x;
                av[4 * v4 + 1] = w4.y;
                av[4 * v4 + 2] = w4.z;
                av[4 * v4 + 3] = w4.w;
              }
#pragma unroll
              for (int q = 0; q < R; ++q)
#pragma unroll
                for (int cc = 0; cc < S; ++cc) acc[q][cc] = fmaf(av[q], b[cc], acc[q][cc]);
            }
          }
          buf ^= 1;
        }
        __syncthreads();                             // every thread is done with Ds
        // new fields and the next change matrix (rows >= Mm are never read)
        const int actm = a.act[m];
        const float gm = a.g[m];
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const int r = ty * R + q;
          if (r < Mm) {
#pragma unroll
            for (int cc = 0; cc < S; ++cc) {
              const int t = tx * S + cc, n = n0 + t;
              const float zo = kAhead ? zf[kAhead ? q : 0][cc] : Zm[(size_t)r * Np + n];
              const float zn = zo + acc[q][cc];
              float d = 0.0f;
              if (n < N && zn != zo) {
                d = hidden_act(actm, zn, gm) - hidden_act(actm, zo, gm);
                if (COMMIT) Zm[(size_t)r * Np + n] = zn;
              }
              if (Sm && n < N) Sm[(size_t)r * Np + n] = zn;
              Ds[r * TS + t] = d;
            }
          }
        }
        __syncthreads();
      }

      // ---- output layer: Z'_{L-1} = Z_{L-1} + W_{L-1} D, loss. The features are cut into
      // 256 / TS parts per sample, added in part order.
      {
        constexpr int PARTS = kDeepThreads / TS;
        const int mo = L - 1;
        const int Ko = a.n_in[mo];
        const float* Wo = a.w[mo];
        const int t = tid % TS, p = tid / TS, n = n0 + t;
        const int per = (Ko + PARTS - 1) / PARTS;
        float s[kMaxC];
#pragma unroll
        for (int q = 0; q < kMaxC; ++q) s[q] = 0.0f;
#pragma unroll 2
        for (int kk = p * per; kk < min(Ko, p * per + per); ++kk) {
          const float d = Ds[kk * TS + t];
#pragma unroll
          for (int q = 0; q < kMaxC; ++q)
            if (q < a.C) s[q] = fmaf(__ldg(Wo + (size_t)q * Ko + kk), d, s[q]);
        }
        __syncthreads();                             // Ds takes the parts
#pragma unroll
        for (int q = 0; q < kMaxC; ++q) Ds[(p * kMaxC + q) * TS + t] = s[q];
        __syncthreads();
        if (p == 0 && n < N) {
          float zz[kMaxC];
          bool changed = false;
#pragma unroll
          for (int q = 0; q < kMaxC; ++q) {
            zz[q] = 0.0f;
            if (q < a.C) {
              float v = 0.0f;
#pragma unroll
              for (int u = 0; u < PARTS; ++u) v += Ds[(u * kMaxC + q) * TS + t];
              const float zo = a.Z[mo][(size_t)q * Np + n];
              zz[q] = zo + v;
              changed |= zz[q] != zo;
            }
          }
          dl = out_delta<COMMIT>(a, n, zz, changed, sk_z, sk_l);
        }
      }
    }
  }
  if (!COMMIT) {
    const float tot = block_sum(dl, s_red);
    if (tid == 0) *part = tot;
  }
}

// One CTA: dS per candidate (fixed order over tiles, compensated fp32), the decision (Eq. 6),
// trace, statistics, and the accepted weight's new value.
__global__ void __launch_bounds__(kKmax) deep_decide_kernel(DeepArgs a) {
  __shared__ DeepCand s_c[kKmax];
  __shared__ float s_dS[kKmax];
  __shared__ int s_take[kKmax];
  __shared__ float s_sum[kKmax];
  __shared__ float s_buf[(kKmax / 32) * 256];
  __shared__ unsigned int s_macc[kKmax / 32], s_mbad[kKmax / 32], s_mforced[kKmax / 32];
  const int k = threadIdx.x, lane = k & 31, warp = k >> 5;
  const int Kb = a.n_explicit > 0 ? a.n_explicit : a.Kb;
  bool acc = false, bad = false, forced = false;
  if (k < Kb) {
    const DeepCand c = deep_candidate(a, k);
    s_c[k] = c;
    s_take[k] = c.valid && c.delta != 0.0f;
  }
  __syncthreads();
  ordered_row_sums(a.partial, a.ntiles, Kb, s_take, s_sum, s_buf);
  if (k < Kb) {
    const DeepCand c = s_c[k];
    const float d = c.valid ? s_sum[k] : __int_as_float(0x7fc00000);
    s_dS[k] = d;
    if (a.n_explicit > 0) {
      a.ex_out[k] = (double)d;
    } else if (c.valid) {
      const unsigned long long tk = a.tau + (unsigned long long)k;
      bool facc = false;
      if (a.nforce > 0) {
        int lo2 = 0, hi2 = a.nforce;
        while (lo2 < hi2) {
          const int mid = (lo2 + hi2) >> 1;
          if (a.ftau[mid] < tk)
            lo2 = mid + 1;
          else
            hi2 = mid;
        }
        if (lo2 < a.nforce && a.ftau[lo2] == tk) {
          forced = true;
          facc = a.facc[lo2] != 0;
        }
      }
      if (forced) {
        acc = facc;
      } else {
        bad = !isfinite(d);
        acc = accept_change(d, a.strict, a.metro, a.seed, tk, a.msc);
      }
    }
  }
  if (a.n_explicit > 0) {
    if (k == 0 && a.ex_tail != nullptr) {
      a.ex_tail->S = a.st->S;
      a.ex_tail->err = a.st->err;
    }
    return;
  }
  const unsigned int ma = __ballot_sync(0xffffffffu, acc);
  const unsigned int mb = __ballot_sync(0xffffffffu, bad);
  const unsigned int mf = __ballot_sync(0xffffffffu, forced);
  if (lane == 0) {
    s_macc[warp] = ma;
    s_mbad[warp] = mb;
    s_mforced[warp] = mf;
  }
  __syncthreads();
  if (k != 0) return;
  int kstar = -1, kbad = -1;
  for (int w = 0; w < kKmax / 32 && kstar < 0; ++w)
    if (s_macc[w]) kstar = w * 32 + __ffs(s_macc[w]) - 1;
  for (int w = 0; w < kKmax / 32 && kbad < 0; ++w)
    if (s_mbad[w]) kbad = w * 32 + __ffs(s_mbad[w]) - 1;
  if (kbad >= 0 && (kstar < 0 || kbad <= kstar)) kstar = -2;
  DevState* st = a.st;
  const int last = kstar >= 0 ? kstar : Kb - 1;
  if (a.trace_cap > 0 && kstar != -2) {
    const double S = st->S;
    for (int q = 0; q <= last; ++q) {
      mca_trace_rec rec;
      rec.tau = a.tau + (unsigned long long)q;
      rec.idx = s_c[q].idx;
      rec.accept = q == kstar ? 1 : 0;
      rec.old_w = s_c[q].oldw;
      rec.new_w = s_c[q].neww;
      rec.valid = s_c[q].valid;
      rec.forced = (int)((s_mforced[q >> 5] >> (q & 31)) & 1u);
      rec.dS = (double)s_dS[q];
      rec.S = S;
      a.trace[st->trace_written % (unsigned long long)a.trace_cap] = rec;
      st->trace_written += 1ull;
    }
  }
  DeepCtl* ctl = a.ctl;
  ctl->kstar = kstar;
  if (kstar == -2) {
    atomicCAS(&st->err, 0, (int)MCA_ERR_NUMERIC);
    ctl->consumed = 0;
    return;
  }
  for (int w = 0; w < kKmax / 32; ++w) {
    unsigned int m = s_mforced[w];
    const int hi = last - w * 32;
    if (hi < 31) m &= hi < 0 ? 0u : ((2u << hi) - 1u);
    if (m) atomicAdd(&st->forced, (unsigned long long)__popc(m));
  }
  // (the statistics below are reductions without a returned value, so this thread does not wait
  // for their reads)
  // FLOPs of the evaluated chains: row update (2 per sample), rank-1 into layer l+1
  // (2 n_out[l+1] per sample), dense layers m = l+2 .. L-1 (2 n_out[m] n_in[m] per sample)
  unsigned long long ncand = 0, flops = 0;
  for (int q = 0; q < Kb; ++q) {
    const DeepCand& c = s_c[q];
    ncand += c.valid ? 1ull : 0ull;
    if (!c.valid || c.delta == 0.0f) continue;
    unsigned long long per = 2ull;
    if (c.layer + 1 < a.L) per += 2ull * (unsigned long long)a.n_out[c.layer + 1];
    for (int m = c.layer + 2; m < a.L; ++m)
      per += 2ull * (unsigned long long)a.n_out[m] * (unsigned long long)a.n_in[m];
    flops += per * (unsigned long long)a.N;
  }
  atomicAdd(&st->candidates, ncand);
  atomicAdd(&st->alg_flops, flops);
  atomicAdd(&st->batches, 1ull);
  if (kstar >= 0) {
    const DeepCand& c = s_c[kstar];
    ctl->acc = c;
    ctl->consumed = kstar + 1;
    atomicAdd(&st->trials, (unsigned long long)(kstar + 1));
    atomicAdd(&st->accepts, 1ull);
    atomicAdd(&st->wasted, (unsigned long long)(Kb - kstar - 1));
    atomicAdd(&st->S, (double)s_dS[kstar]);
    const int l = c.layer;
    const unsigned long long off = c.idx - a.off[l];
    a.w[l][off] = c.neww;
    if (a.wk[l] != MCA_W_FP32) a.code[l][off] = (signed char)c.new_code;
    // split image of the tensor-core chain
    if (a.whi[l] != nullptr) deep_tc_image_store(a, l, c.row, c.col, c.neww);
  } else {
    ctl->consumed = Kb;
    atomicAdd(&st->trials, (unsigned long long)Kb);
  }
}

// Per-sample losses from the output fields, and nothing else (S is summed by sum_loss_kernel).
__global__ void deep_losses_kernel(DeepArgs a) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= a.N) return;
  const int Lo = a.L - 1;
  float zz[kMaxC];
#pragma unroll
  for (int q = 0; q < kMaxC; ++q) zz[q] = q < a.C ? a.Z[Lo][(size_t)q * a.Np + n] : 0.0f;
  a.ell[n] = sample_loss<-1, -1, kMaxC>(zz, a.C, a.y[n], a.g[Lo], a.act[Lo], a.loss);
}

// The SIMT chain's variant: rows per thread from the widest layer behind the first, samples per
// thread from the handle's tile.
using ChainFn = void (*)(DeepArgs);

template <bool COMMIT, int S>
static ChainFn chain_rows(int width, size_t* smem) {
  const int R = width <= 64 ? 4 : width <= 128 ? 8 : 16;
  *smem = sizeof(float) * (size_t)(kDeepMaxWidth * 16 * S + 2 * kDeepKC * 16 * R);
  return R == 4   ? deep_chain_kernel<COMMIT, 4, S>
         : R == 8 ? deep_chain_kernel<COMMIT, 8, S>
                  : deep_chain_kernel<COMMIT, 16, S>;
}

template <bool COMMIT>
static cudaError_t chain_variant(const DeepArgs& a, ChainFn* fn, size_t* smem) {
  int width = 0;
  for (int m = 1; m < a.L - 1; ++m) width = std::max(width, a.n_out[m]);
  *fn = a.tile == 32 ? chain_rows<COMMIT, 2>(width, smem) : chain_rows<COMMIT, 4>(width, smem);
  return cudaFuncSetAttribute((const void*)*fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)*smem);
}

cudaError_t launch_deep_eval(const DeepArgs& a, cudaStream_t s) {
  if (a.tc) return launch_deep_eval_tc(a, s);
  const int Kb = a.n_explicit > 0 ? a.n_explicit : a.Kb;
  ChainFn fn;
  size_t smem;
  cudaError_t e = chain_variant<false>(a, &fn, &smem);
  if (e != cudaSuccess) return e;
  fn<<<dim3(Kb, a.ntiles), kDeepThreads, smem, s>>>(a);
  return cudaGetLastError();
}

// Evaluation CTAs that run at the same time on one SM.
int deep_eval_ctas_per_sm(const DeepArgs& a) {
  if (a.tc) return 1;
  ChainFn fn;
  size_t smem;
  int occ = 0;
  if (chain_variant<false>(a, &fn, &smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kDeepThreads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return std::max(1, occ);
}

cudaError_t launch_deep_decide(const DeepArgs& a, cudaStream_t s) {
  deep_decide_kernel<<<1, kKmax, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_deep_commit(const DeepArgs& a, cudaStream_t s) {
  if (a.tc) return launch_deep_commit_tc(a, s);
  ChainFn fn;
  size_t smem;
  cudaError_t e = chain_variant<true>(a, &fn, &smem);
  if (e != cudaSuccess) return e;
  fn<<<a.ntiles, kDeepThreads, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_deep_losses(const DeepArgs& a, cudaStream_t s) {
  deep_losses_kernel<<<(a.N + 127) / 128, 128, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace mca

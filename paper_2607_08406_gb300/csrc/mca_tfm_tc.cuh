// Pieces shared by the tensor-core Transformer kernels with tf32 operand parts (mca_tfm_tc.cu) and with
// fp16 parts (mca_tfm_f16.cu): the patched parameter read, a candidate's matrix entry and restart key,
// layer-norm statistics, the rank-1 step of a feed-forward hidden unit, and causal attention.
#pragma once

#include <cuda_fp16.h>

#include "mca_device.cuh"
#include "mca_internal.h"
#include "mca_tc.cuh"
#include "mca_tc_layout.h"
#include "mca_tfm.cuh"

namespace mca {
namespace {

constexpr int kRows = 128;                       // token rows per CTA: two sequences
constexpr int kD = kTcTfmD;
constexpr int kT = kTcTfmT;
constexpr int kHc = kTcTfmHc;
constexpr int kXLd = kD + 4;                     // residual row stride: conflict-free row access
constexpr int kTfmWorkers = 512;                 // threads that own token rows

// Barrier of the threads that own token rows (the control warp of the fp16 kernel takes no part).
__device__ __forceinline__ void rows_sync() {
  asm volatile("bar.sync 1, %0;" ::"r"(kTfmWorkers) : "memory");
}

__device__ __forceinline__ float prm(const TfmArgs& a, unsigned long long i,
                                     unsigned long long midx, float mval) {
  return i == midx ? mval : a.params[i];
}

// The weight matrix entry a parameter is (kTcMatNone for biases, LN parameters, embeddings).
struct Target {
  int mat, row, col;
};

__device__ __forceinline__ Target tc_target(const TfmArgs& a, unsigned long long idx, int stage) {
  Target t;
  t.mat = kTcMatNone;
  t.row = 0;
  t.col = 0;
  if (stage >= 0 && stage < a.nL) {
    const unsigned long long off = idx - a.o_blk0 - (unsigned long long)stage * a.blk_size;
    const unsigned long long dd = (unsigned long long)a.d * a.d, fd = (unsigned long long)a.F * a.d;
    const unsigned int rq[4] = {a.r_wq, a.r_wk, a.r_wv, a.r_wo};
#pragma unroll
    for (int m = 0; m < 4; ++m)
      if (off >= rq[m] && off < rq[m] + dd) {
        t.mat = m;
        t.row = (int)((off - rq[m]) / a.d);
        t.col = (int)((off - rq[m]) % a.d);
      }
    if (off >= a.r_w1 && off < a.r_w1 + fd) {
      t.mat = kTcW1;
      t.row = (int)((off - a.r_w1) / a.d);
      t.col = (int)((off - a.r_w1) % a.d);
    }
    if (off >= a.r_w2 && off < a.r_w2 + fd) {
      t.mat = kTcW2;
      t.row = (int)((off - a.r_w2) / a.F);
      t.col = (int)((off - a.r_w2) % a.F);
    }
  } else if (stage == a.nL && idx >= a.o_wh && idx < a.o_wh + (unsigned long long)a.V * a.d) {
    t.mat = kTcHead;
    t.row = (int)((idx - a.o_wh) / a.d);
    t.col = (int)((idx - a.o_wh) % a.d);
  }
  return t;
}

// Where candidate k's recomputation starts, from its proposal alone, as a key that orders the
// recomputations by length: 4 stage, plus 2 for a block's feed-forward sub-block, plus 3 for one of
// its hidden units (then block stage + 1, key 4 stage + 4, follows a short rank-1 step).
__device__ __forceinline__ int candidate_stage(const TfmArgs& a, int k) {
  unsigned int idx;
  if (a.n_explicit > 0) {
    idx = a.ex_idx[k];
  } else {
    const uint4 w = trial_words(a.seed, tfm_batch_tau(a) + (unsigned long long)k);
    idx = (unsigned int)(((unsigned long long)w.x * a.P) >> 32);
  }
  const int st = tfm_stage(a, idx);
  const int rs = tfm_restart(a, idx, st);
  return 4 * st + (rs == kRestartFfn ? 2 : rs == kRestartUnit ? 3 : 0);
}

// What a thread that owns a token row knows.
struct RowCtx {
  float* xs;                 // residual stream [128][kXLd]
  float* ks;                 // K [128][128], 16-byte slots of a row swizzled by (row mod 8)
  float* vs;                 // V, same
  uint32_t tmem;             // tensor-memory base address
  uint32_t trow;             // this warp's lane quarter in a tensor-memory address
  int r, g, sl, t;           // token row, column part, sequence of the pair, position
  unsigned long long midx;   // patched parameter (~0: none)
  float mval, dlt;           // its value, and the change of a weight-matrix entry
  int cstage;                // the stage the candidate feeds (-1 embeddings)
  Target tg;
};

// v[i] += val for the one i == at (none if at is outside the array).
template <int N>
__device__ __forceinline__ void add_at(float (&v)[N], int at, float val) {
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (i == at) v[i] += val;
}

// A candidate in W1, b1, W2 or b2 of block b changes one hidden unit j of the block's feed-forward
// network, so the block's output stream (cached) moves by a rank-1 term: by W2[:, j] (f(u'_j) -
// f(u_j)) for W1[j][k] and b1[j], by delta f(u_j) on column i for W2[i][j], by delta on column i
// for b2[i], with u_j = LN2(mid stream) . W1[j, :] + b1[j] recomputed here on the CUDA cores (the
// candidate's own entry at its old value: in a commit the parameter already holds the new one).
// The new output stream of this thread's row part goes to xr.
__device__ void ffn_unit(const TfmArgs& a, const RowCtx& c, const DeepCand& cd, int s0, float* xr,
                         float* s_part, float* s_acol) {
  const int b = cd.layer;
  const unsigned long long base = a.o_blk0 + (unsigned long long)b * a.blk_size;
  const unsigned long long off = (unsigned long long)cd.idx - base;
  const size_t seq_floats = (size_t)kT * kD;
  int kind, j = 0, i0 = -1, kcol = -1;       // kind: 0 W1[j][kcol], 1 b1[j], 2 W2[i0][j], 3 b2[i0]
  if (off < a.r_b1) {
    kind = 0;
    j = (int)((off - a.r_w1) / kD);
    kcol = (int)((off - a.r_w1) % kD);
  } else if (off < a.r_w2) {
    kind = 1;
    j = (int)(off - a.r_b1);
  } else if (off < a.r_b2) {
    kind = 2;
    i0 = (int)((off - a.r_w2) / (unsigned long long)a.F);
    j = (int)((off - a.r_w2) % (unsigned long long)a.F);
  } else {
    kind = 3;
    i0 = (int)(off - a.r_b2);
  }
  const size_t row = ((size_t)(s0 + c.sl)) * seq_floats + (size_t)c.t * kD + 32 * c.g;
  float xn[32];
  const float* xo = a.X + (size_t)(b + 1) * a.B * seq_floats + row;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 v = reinterpret_cast<const float4*>(xo)[i];
    xn[4 * i] = v.x;
    xn[4 * i + 1] = v.y;
    xn[4 * i + 2] = v.z;
    xn[4 * i + 3] = v.w;
  }
  if (kind == 3) {
    add_at(xn, i0 - 32 * c.g, cd.delta);
  } else {
    float x[32];
    const float* xm = a.Xmid + (size_t)b * a.B * seq_floats + row;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float4 v = reinterpret_cast<const float4*>(xm)[i];
      x[4 * i] = v.x;
      x[4 * i + 1] = v.y;
      x[4 * i + 2] = v.z;
      x[4 * i + 3] = v.w;
    }
    float sm = 0.0f;
#pragma unroll
    for (int i = 0; i < 32; ++i) sm += x[i];
    s_part[c.g * kRows + c.r] = sm;
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
    const unsigned long long w1 = base + a.r_w1 + (unsigned long long)j * kD;
    float p = 0.0f;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const int col = 32 * c.g + i;
      const float ln = (x[i] - mean) * rstd * a.params[base + a.r_ln2g + col] +
                       a.params[base + a.r_ln2b + col];
      if (col == kcol) s_acol[c.r] = ln;
      const float w = w1 + col == cd.idx ? cd.oldw : a.params[w1 + col];
      p = fmaf(ln, w, p);
    }
    s_part[c.g * kRows + c.r] = p;           // every thread has read the means (barrier above)
    rows_sync();
    const float bj = kind == 1 ? cd.oldw : a.params[base + a.r_b1 + j];
    const float u = ((((s_part[c.r] + s_part[kRows + c.r]) + s_part[2 * kRows + c.r]) +
                      s_part[3 * kRows + c.r])) + bj;
    if (kind == 2) {
      add_at(xn, i0 - 32 * c.g, cd.delta * act_rt(a.act, u, a.g));
    } else {
      const float un = kind == 0 ? fmaf(cd.delta, s_acol[c.r], u) : u + cd.delta;
      const float da = act_rt(a.act, un, a.g) - act_rt(a.act, u, a.g);
      const unsigned long long w2 = base + a.r_w2 + (unsigned long long)j;
#pragma unroll
      for (int i = 0; i < 32; ++i)
        xn[i] = fmaf(a.params[w2 + (unsigned long long)(32 * c.g + i) * a.F], da, xn[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
    *reinterpret_cast<float4*>(xr + 4 * i) =
        make_float4(xn[4 * i], xn[4 * i + 1], xn[4 * i + 2], xn[4 * i + 3]);
  rows_sync();                               // s_part and s_acol may be written again
}

// Causal attention of query row r with head g over the keys of its sequence (K and V in shared
// memory), with a running maximum and sum over blocks of 8 keys. The instructions of the warps with 64
// keys bound it, so products come in pairs: an evaluation of the 2-block d_model 128 model on 256
// sequences takes 95.0 us on average, one product at a time 98.9 us.
__device__ __forceinline__ void attention(const RowCtx& c, const float (&q)[32], float (&o)[32]) {
  const float scale = rsqrtf(32.0f);
  const float* kb = c.ks + (size_t)(c.sl * kT) * kD + 32 * c.g;
  const float* vb = c.vs + (size_t)(c.sl * kT) * kD + 32 * c.g;
  float m = -INFINITY, l = 0.0f;
  float2 o2[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) o2[i] = make_float2(0.0f, 0.0f);
  const int jend = (c.t | 31) + 1;               // the same for every lane of the warp
#pragma unroll 1
  for (int j0 = 0; j0 < jend; j0 += 8) {
    float sc[8];
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) {
      const float* kr = kb + (size_t)(j0 + jj) * kD;
      float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 kv = *reinterpret_cast<const float4*>(kr + 4 * (i ^ jj));
        s = fma2(make_float2(q[4 * i], q[4 * i + 1]), make_float2(kv.x, kv.y), s);
        s = fma2(make_float2(q[4 * i + 2], q[4 * i + 3]), make_float2(kv.z, kv.w), s);
      }
      sc[jj] = j0 + jj <= c.t ? (s.x + s.y) * scale : -INFINITY;
    }
    float bm = sc[0];
#pragma unroll
    for (int jj = 1; jj < 8; ++jj) bm = fmaxf(bm, sc[jj]);
    const float mn = fmaxf(m, bm);               // finite: key 0 is in the first block
    const float corr = __expf(m - mn);
    l *= corr;
#pragma unroll
    for (int i = 0; i < 16; ++i) o2[i] = mul2(o2[i], make_float2(corr, corr));
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) {
      const float p = __expf(sc[jj] - mn);
      const float2 p2 = make_float2(p, p);
      l += p;
      const float* vr = vb + (size_t)(j0 + jj) * kD;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 vv = *reinterpret_cast<const float4*>(vr + 4 * (i ^ jj));
        o2[2 * i] = fma2(p2, make_float2(vv.x, vv.y), o2[2 * i]);
        o2[2 * i + 1] = fma2(p2, make_float2(vv.z, vv.w), o2[2 * i + 1]);
      }
    }
    m = mn;
  }
  const float inv = 1.0f / l;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    o[2 * i] = o2[i].x * inv;
    o[2 * i + 1] = o2[i].y * inv;
  }
}

// Weight w, element (r, k) of a matrix, into its image with fp16 parts.
__device__ __forceinline__ void tfm_f16_image_store(const TfmArgs& a, int mat, int b, int r, int k,
                                                    float w) {
  __half* img = reinterpret_cast<__half*>(a.wimg16);
  const size_t o = tfm_f16_image_offset(mat, b, r, k, a.F, a.nL);
  const float x = w * a.f16_w;
  const __half h = __float2half_rn(x);
  img[o] = h;
  img[o + kTfmF16Chunk / 4] = __float2half_rn(x - __half2float(h));
}

// The image entries of the accepted weight-matrix parameter (after the commit kernel, which reads the
// old one).
__device__ __forceinline__ void image_update(const TfmArgs& a, const DeepCand& c) {
  const Target tg = tc_target(a, c.idx, c.layer);
  if (tg.mat == kTcMatNone) return;
  const float w = a.params[c.idx];
  const float hi = tf32_rna(w);
  const size_t o = tfm_tc_image_offset(tg.mat, c.layer, tg.row, tg.col, a.F, a.nL);
  a.wimg[o] = hi;
  a.wimg[o + tc_image_lo(tfm_tc_rows(tg.mat))] = tf32_rna(w - hi);
  tfm_f16_image_store(a, tg.mat, c.layer, tg.row, tg.col, w);
}

}  // namespace
}  // namespace mca

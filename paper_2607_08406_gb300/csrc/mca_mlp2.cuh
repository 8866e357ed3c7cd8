// Trial loop of the single-hidden-layer MCA path (input -> hidden -> output), Section 2.4, as one
// persistent cooperative kernel.
//
// Cached state (feature-major, so that a mutated neuron's field row is contiguous):
//   z1   [H x Np]   hidden local fields z1[j, n] = sum_i W1[j, i] x[n, i]
//   srec [N x 16]   per sample: output fields z2[0..C), the sample's loss, its label
//   X    CSR by input feature: the non-zero entries x[n, i] of feature i, ascending n
//
// A mutation of W1[j, i] changes z1[j, n] by delta * x[n, i] only where x[n, i] != 0 (a rank-1
// update restricted to feature i's non-zeros) and the output fields by W2[:, j] times neuron j's
// activation change. A mutation of W2[o, j] changes z2[o, n] by delta * f(z1[j, n]) for every n.
//
// Work split: the samples are cut into NR contiguous ranges and CTA r owns range r for the whole
// launch -- it is the only CTA that reads or writes z1[:, n] and srec[n] for n in its range, and it
// keeps the range's sample records in shared memory. Per batch of K candidates:
//   propose   every CTA draws all K proposals itself (Philox; no communication)
//   evaluate  each CTA sums l' - l over its own samples for every candidate, in fixed sub-chunks
//             (warp per sub-chunk, fixed lane order), and writes one partial per (candidate, range)
//   barrier   the only grid-wide synchronisation of a batch
//   decide    every CTA sums each candidate's NR partials in the same fixed order and takes the
//             lowest-index candidate with dS <= theta (Eq. 6: theta = 0; Eq. 7: the trial's
//             Metropolis threshold): the same answer in every CTA
//   commit    each CTA applies the accepted candidate to its own samples (no barrier needed: no
//             other CTA reads them) and writes the new weight value (the same value from all CTAs)
// Every partial depends only on (candidate, range), so dS and the trajectory do not depend on K.
#pragma once

#include "mca_device.cuh"
#include "mca_internal.h"

namespace mca {

struct Cand {
  unsigned long long bytes;  // compulsory DRAM bytes of evaluating this candidate (statistics)
  unsigned int idx;
  int layer, row, col;
  float oldw, neww, delta;
  int new_code;
  int valid;
  int gcnt;                  // entries over all samples; 0: nothing changes, dS = 0 exactly
  int ebeg, ecnt;            // this CTA's segment (CSR entries, or samples of the range)
  int sub0, nsub;            // this CTA's sub-chunks
};

__device__ __forceinline__ void fill_candidate(const Mlp2Args& a, unsigned int idx, uint32_t r1,
                                               bool explicit_value, float ex_new, int r, int s0,
                                               int s1, Cand& c) {
  const int layer = (unsigned long long)idx >= a.P1 ? 1 : 0;
  const unsigned long long off = idx - (layer ? a.P1 : 0ull);
  const int n_in = layer ? a.H : a.D;
  c.idx = idx;
  c.layer = layer;
  c.row = (int)((unsigned int)off / (unsigned int)n_in);      // P < 2^32
  c.col = (int)((unsigned int)off % (unsigned int)n_in);
  const Mutation mu = draw_mutation(layer ? a.wk2 : a.wk1, layer ? a.w2 : a.w1,
                                    layer ? a.code2 : a.code1, layer ? a.wfix2 : a.wfix1,
                                    layer ? a.sc2 : a.sc1, off, a.op, a.lo, a.hi, a.delta, a.bound,
                                    r1, explicit_value, ex_new);
  c.oldw = mu.oldw;
  c.neww = mu.neww;
  c.new_code = mu.new_code;
  c.valid = mu.valid;
  c.delta = __fsub_rn(c.neww, c.oldw);
  const int all = layer == 0 ? a.xs_off[c.col + 1] - a.xs_off[c.col] : a.N;
  // A zero change leaves every field bit-identical: dS = 0 exactly, nothing to evaluate.
  c.gcnt = (c.valid && c.delta != 0.0f) ? all : 0;
  c.bytes = 0ull;
  c.ebeg = 0;
  c.ecnt = 0;
  if (c.gcnt > 0) {
    if (layer == 0) {
      const int* ro = a.xs_roff + (size_t)c.col * (a.NR + 1) + r;
      c.ebeg = ro[0];
      c.ecnt = ro[1] - ro[0];
      c.bytes = 32ull * (unsigned long long)a.xs_sect[c.col] + 8ull * (unsigned long long)all;
    } else {
      c.ecnt = s1 - s0;
      c.bytes = 4ull * (unsigned long long)a.N;
    }
  }
  c.nsub = (c.ecnt + a.SUB - 1) / a.SUB;
}

// Sample records of this CTA's range: field f of range-local sample nl at rec[f * pitch + nl].
struct Recs {
  float* rec;
  int pitch;
};

// One entry of a first-layer candidate: range-local sample nl with input value x and cached field
// z; w holds W2[:, j]. Returns l' - l; COMMIT also writes the new hidden field (*zp) and record.
template <int ACT1, int ACT2, int LOSS, int NC, bool COMMIT>
__device__ __forceinline__ float entry_l1(const Mlp2Args& a, Recs R, float delta,
                                          const float (&w)[NC > 0 ? NC : kMaxC], int nl, float x,
                                          float z, float* zp) {
  const float zn = fmaf(delta, x, z);
  const float da = act_compact<ACT1>(zn, a.g1, a.act1) - act_compact<ACT1>(z, a.g1, a.act1);
  if (COMMIT) *zp = zn;
  if (da == 0.0f) return 0.0f;
  constexpr int M = NC > 0 ? NC : kMaxC;
  const int C = NC > 0 ? NC : a.C;
  float zz[M];
  float ell;
  int y;
  load_srec(R.rec, R.pitch, nl, zz, ell, y);
#pragma unroll
  for (int k = 0; k < M; ++k)
    if (k < C) zz[k] = fmaf(w[k], da, zz[k]);
  const float ln = sample_loss<ACT2, LOSS, M, true>(zz, C, y, a.g2, a.act2, a.loss);
  if (COMMIT) store_srec(R.rec, R.pitch, nl, zz, ln, y);
  return ln - ell;
}

// One sample of an output-layer candidate W2[o, j] (o = row, j's cached field z1[j, n] = z).
template <int ACT1, int ACT2, int LOSS, int NC, bool COMMIT>
__device__ __forceinline__ float entry_l2(const Mlp2Args& a, Recs R, float delta, int o, int nl,
                                          float z) {
  constexpr int M = NC > 0 ? NC : kMaxC;
  const int C = NC > 0 ? NC : a.C;
  const float av = act_compact<ACT1>(z, a.g1, a.act1);
  float zz[M];
  float ell;
  int y;
  load_srec(R.rec, R.pitch, nl, zz, ell, y);
  float zo = 0.0f;
#pragma unroll
  for (int k = 0; k < M; ++k)
    if (k == o) zo = zz[k];
  const float zon = fmaf(delta, av, zo);
  if (zon == zo) return 0.0f;
#pragma unroll
  for (int k = 0; k < M; ++k)
    if (k == o) zz[k] = zon;
  const float ln = sample_loss<ACT2, LOSS, M, true>(zz, C, y, a.g2, a.act2, a.loss);
  if (COMMIT) store_srec(R.rec, R.pitch, nl, zz, ln, y);
  return ln - ell;
}

template <int NC>
__device__ __forceinline__ void load_w2c(const float* src, int C, float (&w)[NC > 0 ? NC : kMaxC]) {
  constexpr int M = NC > 0 ? NC : kMaxC;
#pragma unroll
  for (int k = 0; k < M; ++k) w[k] = (NC > 0 || k < C) ? src[k] : 0.0f;
}

// Warp-level sum of l' - l over sub-chunk q of candidate c's segment in this CTA's range. Lane l
// takes entries l, l + 32, ... of the sub-chunk in ascending order (four at a time, loads first).
template <int ACT1, int ACT2, int LOSS, int NC>
__device__ __forceinline__ float eval_sub(const Mlp2Args& a, Recs R, int s0, const Cand& c,
                                          const float* w2c, int q) {
  const int lane = threadIdx.x & 31;
  const int e_lo = q * a.SUB;
  const int e_hi = min(e_lo + a.SUB, c.ecnt);
  const float* zrow = a.z1 + (size_t)(c.layer == 0 ? c.row : c.col) * a.Np;
  const float delta = c.delta;
  const int layer = c.layer, o = c.row, ebeg = c.ebeg;
  float w[NC > 0 ? NC : kMaxC];
  load_w2c<NC>(w2c, a.C, w);
  float acc = 0.0f;
  for (int g = e_lo; g < e_hi; g += 128) {
    int nn[4];
    float xv[4], zv[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int e = g + t * 32 + lane;
      nn[t] = -1;
      xv[t] = 0.0f;
      if (e < e_hi) {
        if (layer == 0) {
          nn[t] = __ldg(a.xs_n + ebeg + e);
          xv[t] = __ldg(a.xs_v + ebeg + e);
        } else {
          nn[t] = s0 + e;
        }
      }
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) zv[t] = nn[t] >= 0 ? zrow[nn[t]] : 0.0f;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (nn[t] < 0) continue;
      if (layer == 0)
        acc += entry_l1<ACT1, ACT2, LOSS, NC, false>(a, R, delta, w, nn[t] - s0, xv[t], zv[t],
                                                     nullptr);
      else
        acc += entry_l2<ACT1, ACT2, LOSS, NC, false>(a, R, delta, o, nn[t] - s0, zv[t]);
    }
  }
  return warp_sum(acc);
}

// Up to four sub-chunks of at most 128 entries each (the common case SUB == 128) at once: every lane
// issues the loads of all its entries (up to 16) before computing any, so one warp keeps up to 512
// gathers in flight. The per-sub-chunk lane order is the same as eval_sub's.
template <int ACT1, int ACT2, int LOSS, int NC>
__device__ __forceinline__ void eval_quad(const Mlp2Args& a, Recs R, int s0, const Cand* cs,
                                          const float (*w2c)[kMaxC], const int (&ks)[4],
                                          const int (&qs)[4], int nq, float (&out)[4]) {
  const int lane = threadIdx.x & 31;
  int nn[16];
  float xv[16], zv[16];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const Cand& c = cs[ks[u]];
    const int e_lo = qs[u] * 128;
    const int e_hi = u < nq ? min(e_lo + 128, c.ecnt) : 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int e = e_lo + t * 32 + lane;
      const int sidx = u * 4 + t;
      nn[sidx] = -1;
      xv[sidx] = 0.0f;
      if (e < e_hi) {
        if (c.layer == 0) {
          nn[sidx] = __ldg(a.xs_n + c.ebeg + e);
          xv[sidx] = __ldg(a.xs_v + c.ebeg + e);
        } else {
          nn[sidx] = s0 + e;
        }
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const Cand& c = cs[ks[u]];
    const float* zrow = a.z1 + (size_t)(c.layer == 0 ? c.row : c.col) * a.Np;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int sidx = u * 4 + t;
      zv[sidx] = nn[sidx] >= 0 ? zrow[nn[sidx]] : 0.0f;
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const Cand& c = cs[ks[u]];
    const float delta = c.delta;
    const int layer = c.layer, o = c.row;
    float w[NC > 0 ? NC : kMaxC];
    load_w2c<NC>(w2c[ks[u]], a.C, w);
    float acc = 0.0f;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int sidx = u * 4 + t;
      if (nn[sidx] < 0) continue;
      if (layer == 0)
        acc += entry_l1<ACT1, ACT2, LOSS, NC, false>(a, R, delta, w, nn[sidx] - s0, xv[sidx],
                                                     zv[sidx], nullptr);
      else
        acc += entry_l2<ACT1, ACT2, LOSS, NC, false>(a, R, delta, o, nn[sidx] - s0, zv[sidx]);
    }
    out[u] = warp_sum(acc);
  }
}

template <int ACT1, int ACT2, int LOSS, int NC>
__global__ void __launch_bounds__(kLoopThreads, 1) mlp2_trial_loop(Mlp2Args a) {
  extern __shared__ __align__(16) float s_records[];
  __shared__ Cand s_c[kKmax];
  __shared__ float s_w2c[kKmax][kMaxC];
  __shared__ float s_sub[kKmax * kMaxSubs];
  __shared__ float s_dS[kKmax];
  __shared__ unsigned int s_macc[kKmax / 32], s_mbad[kKmax / 32], s_mforced[kKmax / 32];
  __shared__ int s_flag, s_kstar, s_total, s_bvalid;
  __shared__ unsigned long long s_bbytes, s_tau_hi;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r = blockIdx.x;
  const int s0 = min(r * a.RS, a.N), s1 = min(s0 + a.RS, a.N);
  const bool explicit_mode = a.n_explicit > 0;
  const Recs R = a.smem_records ? Recs{s_records, a.RS} : Recs{a.srec + s0, a.Np};
  if (a.smem_records) {
    const int ns = s1 - s0;
    for (int t = tid; t < kRecFields * ns; t += kLoopThreads) {
      const int f = t / ns, nl = t - f * ns;
      s_records[f * a.RS + nl] = a.srec[(size_t)f * a.Np + s0 + nl];
    }
  }

  // CTA 0, thread 0 carries the run statistics in registers for the whole launch.
  DevState* st = a.st;
  const bool stats_thread = r == 0 && tid == 0;
  double S = 0.0;
  unsigned long long n_trials = 0, n_acc = 0, n_cand = 0, n_batch = 0, n_waste = 0, n_forced = 0,
                     n_bytes = 0, n_trace = 0, ph0 = 0, ph1 = 0, ph2 = 0, ph3 = 0;
  if (stats_thread) {
    S = st->S;
    n_trace = st->trace_written;
  }
  unsigned int gen = 0;
  unsigned long long tau = a.tau0;
  if (tid == 0) s_tau_hi = a.tau0;
  // acceptance-rate estimate behind the batch width: the same in every CTA
  float rate_a = st->rate_acc, rate_t = st->rate_trials;
  const unsigned long long end = a.tau0 + a.n_trials;
  int buf = 0;
  __syncthreads();

  while (explicit_mode || tau < end) {
    const unsigned long long t_a = stats_thread ? globaltimer_ns() : 0ull;
    const int Kw = a.fixed_K ? a.K : batch_width(rate_a, rate_t, kWidthMlp2, a.K);
    const int Kb = explicit_mode ? a.n_explicit
                                 : (int)((end - tau) < (unsigned long long)Kw ? (end - tau) : Kw);
    // ---- propose: every CTA draws every candidate
    for (int k = tid; k < Kb; k += kLoopThreads) {
      Cand c;
      if (explicit_mode) {
        fill_candidate(a, a.ex_idx[k], 0u, true, a.ex_new[k], r, s0, s1, c);
      } else {
        const uint4 w = trial_words(a.seed, tau + (unsigned long long)k);
        const unsigned int idx =
            mlp2_trial_index(a.P, a.P1, a.seed, tau + (unsigned long long)k, w.x, a.stretch);
        fill_candidate(a, idx, w.y, false, 0.0f, r, s0, s1, c);
      }
      if (c.layer == 0 && c.gcnt > 0) {
#pragma unroll
        for (int q = 0; q < kMaxC; ++q)
          s_w2c[k][q] = q < a.C ? a.w2[(size_t)q * a.H + c.row] : 0.0f;
      }
      s_c[k] = c;
    }
    __syncthreads();
    if (warp == 0) {                 // exclusive scan of the sub-chunk counts; batch statistics
      int v[4], loc = 0;
      unsigned long long bytes = 0ull;
      int valid = 0;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int k = lane * 4 + t;
        v[t] = k < Kb ? s_c[k].nsub : 0;
        loc += v[t];
        if (k < Kb) {
          // bytes of candidates not evaluated before in this launch (a candidate re-evaluated in
          // the next batch finds its data on chip)
          if (tau + (unsigned long long)k >= s_tau_hi) bytes += s_c[k].bytes;
          valid += s_c[k].valid;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        bytes += __shfl_xor_sync(0xffffffffu, bytes, o);
        valid += __shfl_xor_sync(0xffffffffu, valid, o);
      }
      if (lane == 0) {
        s_bbytes = bytes;
        s_bvalid = valid;
      }
      int inc = loc;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      int ex = inc - loc;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int k = lane * 4 + t;
        if (k < Kb) s_c[k].sub0 = ex;
        ex += v[t];
      }
      if (lane == 31) s_total = inc;
    }
    __syncthreads();

    // ---- evaluate this CTA's samples: warp per sub-chunk (four at a time when SUB == 128)
    {
      const int total = s_total;
      int k = 0;
      if (a.SUB == 128) {
        for (int it0 = warp; it0 < total; it0 += 4 * kLoopWarps) {
          int ks[4], qs[4], nq = 0;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int it = it0 + u * kLoopWarps;
            ks[u] = k;
            qs[u] = 0;
            if (it < total) {
              while (s_c[k].sub0 + s_c[k].nsub <= it) ++k;
              ks[u] = k;
              qs[u] = it - s_c[k].sub0;
              nq = u + 1;
            }
          }
          float v[4];
          eval_quad<ACT1, ACT2, LOSS, NC>(a, R, s0, s_c, s_w2c, ks, qs, nq, v);
          if (lane == 0) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (u < nq) s_sub[it0 + u * kLoopWarps] = v[u];
          }
        }
      } else {
        for (int it = warp; it < total; it += kLoopWarps) {
          while (s_c[k].sub0 + s_c[k].nsub <= it) ++k;
          const float v =
              eval_sub<ACT1, ACT2, LOSS, NC>(a, R, s0, s_c[k], s_w2c[k], it - s_c[k].sub0);
          if (lane == 0) s_sub[it] = v;
        }
      }
    }
    __syncthreads();
    float* part = a.partial + (size_t)buf * kKmax * a.NR;
    for (int k = tid; k < Kb; k += kLoopThreads) {
      float s = 0.0f;
      const int b = s_c[k].sub0, nb = s_c[k].nsub;
      for (int q = 0; q < nb; ++q) s += s_sub[b + q];
      part[(size_t)k * a.NR + r] = s;
    }
    const unsigned long long t_b = stats_thread ? globaltimer_ns() : 0ull;
    if (!grid_sync(a.bar, gridDim.x, gen, &st->err, &s_flag)) break;
    const unsigned long long t_c = stats_thread ? globaltimer_ns() : 0ull;

    // ---- dS of every candidate: the NR partials in a fixed order (lane-strided, compensated
    // fp32). A warp takes candidates warp, warp + 16, warp + 32, warp + 48 together, loads first.
    for (int k0 = warp; k0 < Kb; k0 += 4 * kLoopWarps) {
      float hi[4] = {0.0f, 0.0f, 0.0f, 0.0f}, lo[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      for (int q0 = 0; q0 < a.NR; q0 += 32 * 8) {
        float v[4][8];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int k = k0 + u * kLoopWarps;
          const bool live = k < Kb && s_c[k].gcnt > 0;
#pragma unroll
          for (int m = 0; m < 8; ++m) {
            const int q = q0 + m * 32 + lane;
            v[u][m] = (live && q < a.NR) ? part[(size_t)k * a.NR + q] : 0.0f;
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int m = 0; m < 8; ++m) two_sum_add(hi[u], lo[u], v[u][m]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int k = k0 + u * kLoopWarps;
        const float t = warp_sum_comp(hi[u], lo[u]);
        if (lane == 0 && k < Kb) s_dS[k] = s_c[k].valid ? t : __int_as_float(0x7fc00000);
      }
    }
    __syncthreads();
    if (explicit_mode) {
      if (r == 0)
        for (int k = tid; k < Kb; k += kLoopThreads) a.ex_out[k] = (double)s_dS[k];
      break;
    }

    // ---- decide (the same in every CTA): lowest-index candidate with dS <= theta (Eq. 6 / 7)
    if (warp < kKmax / 32) {
      bool acc = false, bad = false, forced = false;
      const int k = tid;
      if (k < Kb && s_c[k].valid) {
        const unsigned long long tk = tau + (unsigned long long)k;
        bool facc = false;
        if (a.nforce > 0) {          // binary search of the forced-decision list
          int lo = 0, hi = a.nforce;
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (a.ftau[mid] < tk)
              lo = mid + 1;
            else
              hi = mid;
          }
          if (lo < a.nforce && a.ftau[lo] == tk) {
            forced = true;
            facc = a.facc[lo] != 0;
          }
        }
        const float d = s_dS[k];
        if (forced) {
          acc = facc;
        } else {
          bad = !isfinite(d);
          acc = accept_change(d, a.strict, a.metro, a.seed, tk, a.msc);
        }
      }
      const unsigned int ma = __ballot_sync(0xffffffffu, acc);
      const unsigned int mb = __ballot_sync(0xffffffffu, bad);
      const unsigned int mf = __ballot_sync(0xffffffffu, forced);
      if (lane == 0) {
        s_macc[warp] = ma;
        s_mbad[warp] = mb;
        s_mforced[warp] = mf;
      }
    }
    __syncthreads();
    if (tid == 0) {
      int kstar = -1, kbad = -1;
      for (int w = 0; w < kKmax / 32 && kstar < 0; ++w)
        if (s_macc[w]) kstar = w * 32 + __ffs(s_macc[w]) - 1;
      for (int w = 0; w < kKmax / 32 && kbad < 0; ++w)
        if (s_mbad[w]) kbad = w * 32 + __ffs(s_mbad[w]) - 1;
      if (kbad >= 0 && (kstar < 0 || kbad <= kstar)) kstar = -2;
      s_kstar = kstar;
      if (stats_thread) {
        const int last = kstar >= 0 ? kstar : Kb - 1;
        if (a.trace_cap > 0) {
          for (int k = 0; k <= last; ++k) {
            mca_trace_rec rec;
            rec.tau = tau + (unsigned long long)k;
            rec.idx = s_c[k].idx;
            rec.accept = k == kstar ? 1 : 0;
            rec.old_w = s_c[k].oldw;
            rec.new_w = s_c[k].neww;
            rec.valid = s_c[k].valid;
            rec.forced = (int)((s_mforced[k >> 5] >> (k & 31)) & 1u);
            rec.dS = (double)s_dS[k];
            rec.S = S;
            a.trace[n_trace % (unsigned long long)a.trace_cap] = rec;
            ++n_trace;
          }
        }
        for (int w = 0; w < kKmax / 32; ++w) {
          unsigned int m = s_mforced[w];
          const int hi = last - w * 32;
          if (hi < 31) m &= hi < 0 ? 0u : ((2u << hi) - 1u);
          n_forced += (unsigned long long)__popc(m);
        }
        n_cand += (unsigned long long)s_bvalid;
        n_bytes += s_bbytes;
        ++n_batch;
        if (kstar >= 0) {
          n_trials += (unsigned long long)(kstar + 1);
          ++n_acc;
          n_waste += (unsigned long long)(Kb - kstar - 1);
          S += (double)s_dS[kstar];
          if (s_c[kstar].layer == 0 && s_c[kstar].gcnt > 0)
            n_bytes += 32ull * (unsigned long long)a.xs_sect[s_c[kstar].col];
        } else if (kstar == -1) {
          n_trials += (unsigned long long)Kb;
        }
      }
    }
    __syncthreads();
    const int kstar = s_kstar;
    const unsigned long long t_d = stats_thread ? globaltimer_ns() : 0ull;
    if (kstar == -2) {                // the same non-finite candidate in every CTA
      if (stats_thread) atomicCAS(&st->err, 0, (int)MCA_ERR_NUMERIC);
      break;
    }

    // ---- commit the accepted candidate to this CTA's samples (no writes on a reject)
    if (kstar >= 0) {
      const Cand& c = s_c[kstar];
      if (c.gcnt > 0) {
        if (c.layer == 0) {
          float* zrow = a.z1 + (size_t)c.row * a.Np;
          float w[NC > 0 ? NC : kMaxC];
          load_w2c<NC>(s_w2c[kstar], a.C, w);
          for (int e = tid; e < c.ecnt; e += kLoopThreads) {
            const int n = __ldg(a.xs_n + c.ebeg + e);
            const float x = __ldg(a.xs_v + c.ebeg + e);
            (void)entry_l1<ACT1, ACT2, LOSS, NC, true>(a, R, c.delta, w, n - s0, x, zrow[n],
                                                      zrow + n);
          }
        } else {
          const float* zrow = a.z1 + (size_t)c.col * a.Np;
          for (int e = tid; e < c.ecnt; e += kLoopThreads)
            (void)entry_l2<ACT1, ACT2, LOSS, NC, true>(a, R, c.delta, c.row, e, zrow[s0 + e]);
        }
      }
      if (tid == 0) {                 // every CTA writes the same value
        const unsigned long long off = c.idx - (c.layer ? a.P1 : 0ull);
        (c.layer ? a.w2 : a.w1)[off] = c.neww;
        const int wk = c.layer ? a.wk2 : a.wk1;
        if (wk != MCA_W_FP32) (c.layer ? a.code2 : a.code1)[off] = (signed char)c.new_code;
      }
      __syncthreads();
      if (tid == 0) s_tau_hi = max(s_tau_hi, tau + (unsigned long long)Kb);
      tau += (unsigned long long)(kstar + 1);
      rate_a = rate_a * kRateDecay + 1.0f;
      rate_t = rate_t * kRateDecay + (float)(kstar + 1);
    } else {
      if (tid == 0) s_tau_hi = max(s_tau_hi, tau + (unsigned long long)Kb);
      tau += (unsigned long long)Kb;
      rate_a = rate_a * kRateDecay;
      rate_t = rate_t * kRateDecay + (float)Kb;
    }
    if (stats_thread) {
      const unsigned long long t_e = globaltimer_ns();
      ph0 += t_b - t_a;
      ph1 += t_c - t_b;
      ph2 += t_d - t_c;
      ph3 += t_e - t_d;
    }
    buf ^= 1;
  }

  // ---- epilogue: sample records back to global memory, statistics to the device state
  if (a.smem_records && !explicit_mode) {
    __syncthreads();
    const int ns = s1 - s0;
    for (int t = tid; t < kRecFields * ns; t += kLoopThreads) {
      const int f = t / ns, nl = t - f * ns;
      a.srec[(size_t)f * a.Np + s0 + nl] = s_records[f * a.RS + nl];
    }
  }
  if (stats_thread && explicit_mode && a.ex_tail != nullptr) {
    a.ex_tail->S = st->S;
    a.ex_tail->err = st->err;
  }
  if (stats_thread && !explicit_mode) {
    st->S = S;
    st->trials += n_trials;
    st->accepts += n_acc;
    st->candidates += n_cand;
    st->batches += n_batch;
    st->wasted += n_waste;
    st->forced += n_forced;
    st->alg_bytes += n_bytes;
    st->trace_written = n_trace;
    st->phase_ns[0] += ph0;
    st->phase_ns[1] += ph1;
    st->phase_ns[2] += ph2;
    st->phase_ns[3] += ph3;
    st->rate_acc = rate_a;
    st->rate_trials = rate_t;
  }
}

// ------------------------------------------------------------------------------------------------
// Windowed trial loop. Same work split, order of sums and decisions as mlp2_trial_loop, but each CTA
// keeps a ring of kWS candidate slots: slot (t mod kWS) holds trial t's candidate for this CTA's range
// and, for first-layer candidates with at most kCap entries in the range, the gathered entries
// (range-local sample, activation change f(z + delta x) - f(z), new field z + delta x). A batch then
// evaluates and commits from shared memory only.
//
// The CTA's warps have two roles. kProdWarps producer warps prepare slots ahead of the batches
// (Philox, weight, CSR and z1 gathers), in trial order, never more than kWS trials ahead; they take
// no part in the batch's barriers, so their memory latency overlaps everything else. The other
// (consumer) warps run the batches: set-up, evaluation, the grid-wide exchange, decision, commit.
// A slot records how many commits this CTA had made when its preparation began (its epoch); every
// commit is appended to a log. Before a batch uses a slot, the log entries since its epoch are
// replayed: a commit of the same weight (its old value changed) or of a first-layer weight on the
// same hidden row (z1 changed) sends the slot back for preparation; a commit of its W2 column is
// patched in. Three consumer warps look at the slots ahead once per batch, one lane per slot: they
// replay the log, send stale slots back to the producers and note which slots are ready and live, so
// that the next batch's set-up only checks its slots against the commit that is still pending. (With
// 64 hidden neurons every second slot goes stale before its batch; prepared again by the batch itself,
// one after another, that took 8.9 us per batch, against 3.6.)
//
// In the first thousands of trials a batch takes 3.3 to 3.9 us by network; in trials 200k to 1M of
// 784-16384-10 on 60000 samples (29 % accepted, six candidates) 4.1 us. Time stamps of a batch of
// that net near its start (an instrumented build; us since the first CTA began it): set-up and
// commit done 1.05, barrier 1.37, the warps know their chunks 1.68, last chunk 2.62, shares added 2.92, next batch
// 4.78. The last step, the slowest CTA's share reaching L2, the poll, the decision and two barriers, is the
// longest. Inside, registers are the limit: variants that spill a hundred bytes are 5 to 10 % slower.
// ------------------------------------------------------------------------------------------------
struct WSlot {
  Cand c;
  unsigned long long ticket;  // trial + 1 once the slot is ready for it (written last)
  int state;                  // 1 entries cached (or nothing to evaluate), 2 read from global
  int epoch;                  // commits of this CTA before the slot's data were read
  float theta;                // the trial's acceptance threshold (Eq. 6: 0; Eq. 7)
};

// One logged commit of the windowed loop.
struct CommitLog {
  unsigned int idx;
  int layer, row, col;
  float neww;
  int changes_z1;             // a first-layer commit with entries: its z1 row changed
};

// Per-phase device timers of the windowed loop (statistics only; each read of the global timer
// sits on the batch's critical path). Built in with -DMCA_PHASE_TIMERS=1.
#ifndef MCA_PHASE_TIMERS
#define MCA_PHASE_TIMERS 0
#endif
constexpr bool kPhaseTimers = MCA_PHASE_TIMERS != 0;
constexpr int kLogLen = 128;
static_assert(kCap <= 32 * kMaxSubs, "chunks of a cached candidate");
static_assert(kLogLen > kWS, "a slot is used at most kWS commits after its preparation began");
// Trials the producers may prepare past the oldest slot in use, for a batch of Kb candidates. Every
// first-layer commit makes 1 / H of the prepared slots stale (the same hidden row), so small layers
// keep the producers close; they must stay far enough ahead to hide one preparation.
__device__ __forceinline__ int window_lead(int H, int Kb) {
  return min(kWS, max(Kb + 24, H / 8));
}
// The first of the three consumer warps that look at the slots ahead (one lane per slot).
constexpr int kLookWarp0 = kLoopWarps - 3 - kWS / 32;
constexpr int kRedoLen = 128;
static_assert(kRedoLen >= kWS, "every slot may be waiting for its second preparation");
constexpr int kProdWarps = 3;
constexpr int kConsWarps = kLoopWarps - kProdWarps;
static_assert(kLookWarp0 == kConsWarps - kWS / 32 && kWS % 32 == 0, "one lane per slot");
constexpr int kConsThreads = kConsWarps * 32;

// Warps per candidate when a batch has n live ones (n = x + 1; the last entry serves any larger n), four
// bits each, and ceil(256 / those), nine bits each: v / w = (v ceil(256 / w)) / 256 for v < kConsWarps.
constexpr int kWpcLast = kConsWarps / 2;
constexpr int warps_per_cand(int x) { return x < kWpcLast ? kConsWarps / (x + 1) : 1; }
constexpr unsigned long long wpc_table(int bits, bool inverse) {
  unsigned long long t = 0;
  for (int x = 0; x <= kWpcLast; ++x) {
    const int w = warps_per_cand(x);
    t |= (unsigned long long)(inverse ? (256 + w - 1) / w : w) << (bits * x);
  }
  return t;
}
constexpr bool wpc_exact() {
  for (int x = 0; x <= kWpcLast; ++x)
    for (int v = 0; v < kConsWarps; ++v) {
      const int w = warps_per_cand(x);
      if (((v * ((256 + w - 1) / w)) >> 8) != v / w) return false;
    }
  return true;
}
constexpr unsigned long long kWpc = wpc_table(4, false), kWpcInv = wpc_table(9, true);
static_assert(9 * (kWpcLast + 1) <= 64 && kConsWarps < 16 && wpc_exact(), "warp split tables");

// Place of the i-th set bit of a mask (a whole warp).
__device__ __forceinline__ int nth_bit(unsigned long long mask, int i) {
  const int lane = threadIdx.x & 31;
  const unsigned int lt = (1u << lane) - 1u;
  const unsigned int l0 = (unsigned int)mask, l1 = (unsigned int)(mask >> 32);
  const int n0 = __popc(l0);
  const unsigned int half = i < n0 ? l0 : l1;
  const int rank = i < n0 ? i : i - n0;
  const unsigned int hit = __ballot_sync(
      0xffffffffu, ((half >> lane) & 1u) != 0u && __popc(half & lt) == rank);
  return __ffs(hit) - 1 + (i < n0 ? 0 : 32);
}

// Barrier of the consumer warps only (named barrier 1).
__device__ __forceinline__ void cons_sync() {
  asm volatile("bar.sync 1, %0;" ::"r"(kConsThreads) : "memory");
}

inline size_t window_smem_bytes(int RS) {
  return sizeof(float) * (size_t)kRecFields * RS +
         (size_t)kWS * kCap * (sizeof(unsigned short) + 2 * sizeof(float));
}

// ------------------------------------------------------------------------------------------------
// Sample records of the windowed loop, and the change of one sample. What bounds a batch is the number
// of instructions that one warp has to execute one after another, so a record is a vector per sample
// (read with three or four 16-byte loads), output fields come in pairs (one instruction for two), and
// the fields past the class count hold -infinity, whose exponential and sigmoid are 0, instead of a
// test per field. (A batch of 391-1001-7 masked nets with MSE on 12347 samples: 4.50 us with one 4-byte load
// and one instruction per field, 3.70 with vectors, all else as it was then.)
//
// M = 10 fields (up to 10 classes): 12 floats a sample, M = 14: 16 floats whose 16-byte parts are
// permuted by the sample's number, so that the lanes of a warp, which read different samples, spread
// over the banks (12 floats do by themselves). The loss and the label follow the fields.
// ------------------------------------------------------------------------------------------------
template <int M>
struct VRecs {
  static_assert(M == 10 || M == 14, "record sizes");
  static constexpr int kStride = M + 2;
  float* rec;
  __device__ __forceinline__ float* part(int n, int q) const {
    return rec + n * kStride + 4 * (M == 10 ? q : q ^ ((n >> 1) & 3));
  }
  __device__ __forceinline__ float& at(int n, int f) const { return part(n, f >> 2)[f & 3]; }
  __device__ __forceinline__ void load(int n, float2 (&z)[M / 2], float& ell, int& y) const {
#pragma unroll
    for (int q = 0; q < kStride / 4; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(part(n, q));
      z[2 * q] = make_float2(v.x, v.y);
      if (2 * q + 1 < M / 2) {
        z[2 * q + 1] = make_float2(v.z, v.w);
      } else {
        ell = v.z;
        y = __float_as_int(v.w);
      }
    }
  }
  __device__ __forceinline__ void store(int n, const float2 (&z)[M / 2], float ell, int y) const {
#pragma unroll
    for (int q = 0; q < kStride / 4; ++q) {
      const bool last = 2 * q + 1 == M / 2;
      const float2 b = last ? make_float2(ell, __int_as_float(y)) : z[last ? 0 : 2 * q + 1];
      *reinterpret_cast<float4*>(part(n, q)) = make_float4(z[2 * q].x, z[2 * q].y, b.x, b.y);
    }
  }
};

// Loss of the fields z with label y; zy: field y; onehot: -[k == y] per field (MSE). The same operations on
// each field and the same order of sums as sample_loss with PAIRS, which the forward pass calls.
template <int ACT2, int LOSS, int M>
__device__ __forceinline__ float vloss(const Mlp2Args& a, const float2 (&z)[M / 2], int y, float zy,
                                       const float* onehot) {
  if constexpr (ACT2 == MCA_ACT_IDENTITY && LOSS == MCA_LOSS_SOFTMAX_CE) {
    float m = fmaxf(z[0].x, z[0].y);
#pragma unroll
    for (int q = 1; q < M / 2; ++q) m = fmaxf(m, fmaxf(z[q].x, z[q].y));
    float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int q = 0; q < M / 2; ++q) {
      const float2 t = mul2(add2(z[q], make_float2(-m, -m)), make_float2(kLog2e, kLog2e));
      s = add2(s, make_float2(ex2_ftz(t.x), ex2_ftz(t.y)));
    }
    return ce_loss(m, s.x + s.y, zy);
  } else if constexpr (ACT2 == MCA_ACT_SIGMOID && LOSS == MCA_LOSS_MSE_ONEHOT) {
    const float* oh = onehot + 16 * y;
    float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int q = 0; q < M / 2; ++q) {
      const float2 t = mul2(z[q], make_float2(-kLog2e, -kLog2e));
      const float2 u = add2(make_float2(ex2_ftz(t.x), ex2_ftz(t.y)), make_float2(1.0f, 1.0f));
      const float2 d = add2(make_float2(rcp_ftz(u.x), rcp_ftz(u.y)),
                            *reinterpret_cast<const float2*>(oh + 2 * q));
      s = fma2(d, d, s);
    }
    return s.x + s.y;
  } else {
    float zz[M];
#pragma unroll
    for (int q = 0; q < M / 2; ++q) {
      zz[2 * q] = z[q].x;
      zz[2 * q + 1] = z[q].y;
    }
    return sample_loss<-1, -1, M, true>(zz, a.C, y, a.g2, a.act2, a.loss);
  }
}

// The direction in which a candidate moves the output fields, per unit of its entries' numbers:
// W2[:, j] for a first-layer weight (w2c), delta on field o for an output-layer weight W2[o, j].
template <int M>
struct Direction {
  float2 w[M / 2];
  const float* w2c;          // first layer: the column, in shared memory
  int o;                     // output layer: the field (-1: first layer)
  float delta;
  __device__ __forceinline__ float at(int y) const { return o < 0 ? w2c[y] : y == o ? delta : 0.0f; }
};

template <int M>
__device__ __forceinline__ Direction<M> direction(const Cand& c, const float* w2c) {
  Direction<M> d;
  d.w2c = w2c;
  d.o = c.layer == 0 ? -1 : c.row;
  d.delta = c.delta;
#pragma unroll
  for (int q = 0; q < M / 2; ++q)
    d.w[q] = c.layer == 0 ? *reinterpret_cast<const float2*>(w2c + 2 * q)
                          : make_float2(2 * q == c.row ? c.delta : 0.0f,
                                        2 * q + 1 == c.row ? c.delta : 0.0f);
  return d;
}

// The change of a sample whose activation change is not finite: 0 times it is no change of the fields
// that the candidate does not touch. (A call: the same inline took 2 % of every batch.)
template <int M, bool COMMIT>
__device__ __noinline__ float vdelta_any(const Mlp2Args& a, VRecs<M> R, const float* w2c, int o,
                                         float delta, int nl, float da) {
  float zz[M];
#pragma unroll
  for (int f = 0; f < M; ++f) {
    const float z = R.at(nl, f);
    zz[f] = o >= 0 ? (f == o ? fmaf(delta, da, z) : z) : f < a.C ? fmaf(w2c[f], da, z) : z;
  }
  const float ell = R.at(nl, M);
  const float ln = sample_loss<-1, -1, M, true>(zz, a.C, __float_as_int(R.at(nl, M + 1)), a.g2, a.act2,
                                          a.loss);
  if (COMMIT) {
#pragma unroll
    for (int f = 0; f < M; ++f) R.at(nl, f) = zz[f];
    R.at(nl, M) = ln;
  }
  return ln - ell;
}

// l' - l of sample nl whose fields move by da along dir; COMMIT also writes the new record (not when
// nothing changes). Exactly 0 when da == 0, or when an output-layer weight moves no field.
template <int ACT2, int LOSS, int M, bool COMMIT>
__device__ __forceinline__ float vdelta(const Mlp2Args& a, const VRecs<M>& R, const float* onehot,
                                        const Direction<M>& dir, int nl, float da) {
  if (!(fabsf(da) < INFINITY))
    return vdelta_any<M, COMMIT>(a, R, dir.w2c, dir.o, dir.delta, nl, da);
  float2 z[M / 2];
  float ell;
  int y;
  R.load(nl, z, ell, y);
  const float zy = LOSS == MCA_LOSS_SOFTMAX_CE ? fmaf(dir.at(y), da, R.at(nl, y)) : 0.0f;
  bool same = da == 0.0f;
  if (dir.o >= 0) {
    const float zo = R.at(nl, dir.o);
    same = fmaf(dir.delta, da, zo) == zo;
  }
#pragma unroll
  for (int q = 0; q < M / 2; ++q) z[q] = fma2(dir.w[q], make_float2(da, da), z[q]);
  const float ln = vloss<ACT2, LOSS, M>(a, z, y, zy, onehot);
  if (COMMIT && !same) R.store(nl, z, ln, y);
  return same ? 0.0f : ln - ell;
}

// The vector W2[:, j] of a first-layer candidate.
template <int M>
__device__ __forceinline__ void load_column(const float* w2c, float2 (&w)[M / 2]) {
#pragma unroll
  for (int q = 0; q < M / 2; ++q) w[q] = *reinterpret_cast<const float2*>(w2c + 2 * q);
}

// l' - l of cached entry e of a slot (of n), for first-layer candidates (only they are cached); z, ln: the new
// fields and loss of its sample nl with label y.
template <int ACT2, int LOSS, int M>
__device__ __forceinline__ float cached_entry(const Mlp2Args& a, const VRecs<M>& R,
                                              const float* onehot, const float2 (&w)[M / 2],
                                              const float* w2c, const unsigned short* nls,
                                              const float* das, int e, int n, float2 (&z)[M / 2],
                                              float& ln, int& nl, int& y) {
  nl = e < n ? (int)nls[e] : 0;
  const float d = e < n ? das[e] : 0.0f;
  float ell;
  R.load(nl, z, ell, y);
  const float zy = LOSS == MCA_LOSS_SOFTMAX_CE ? fmaf(w2c[y], d, R.at(nl, y)) : 0.0f;
#pragma unroll
  for (int q = 0; q < M / 2; ++q) z[q] = fma2(w[q], make_float2(d, d), z[q]);
  ln = vloss<ACT2, LOSS, M>(a, z, y, zy, onehot);
  return d == 0.0f ? 0.0f : ln - ell;
}

// Commit of cached entry e whose new loss ln is known: the record and the hidden field.
template <int M>
__device__ __forceinline__ void commit_entry(const VRecs<M>& R, const float2 (&w)[M / 2],
                                             const unsigned short* nls, const float* das,
                                             const float* zns, int e, float ln, float* zrow) {
  const int nl = nls[e];
  const float d = das[e];
  zrow[nl] = zns[e];
  if (d == 0.0f) return;
  float2 z[M / 2];
  float ell;
  int y;
  R.load(nl, z, ell, y);
#pragma unroll
  for (int q = 0; q < M / 2; ++q) z[q] = fma2(w[q], make_float2(d, d), z[q]);
  R.store(nl, z, ln, y);
}

// The number that goes with an entry, from global memory: f(z + delta x) - f(z) (zn = z + delta x), or
// f(z) for an output-layer weight.
template <int ACT1>
__device__ __forceinline__ float entry_step(const Mlp2Args& a, const Cand& c, float x, float z,
                                            float& zn) {
  const float f = act_compact<ACT1>(z, a.g1, a.act1);
  zn = z;
  if (c.layer != 0) return f;
  zn = fmaf(c.delta, x, z);
  return act_compact<ACT1>(zn, a.g1, a.act1) - f;
}

// Warp-level sum of l' - l over chunk q (of a.SUB entries) of a candidate that is not cached. Lane l
// takes entries l, l + 32, ... in ascending order; the next entry's loads are in flight.
template <int ACT1, int ACT2, int LOSS, int M>
__device__ __forceinline__ float eval_global(const Mlp2Args& a, const VRecs<M> R,
                                             const float* onehot, int s0, const Cand& c,
                                             const float* w2c, int q) {
  const int e_hi = min(q * a.SUB + a.SUB, c.ecnt);
  const float* zrow = a.z1 + (size_t)(c.layer == 0 ? c.row : c.col) * a.Np;
  const Direction<M> dir = direction<M>(c, w2c);
  float acc = 0.0f, x1 = 0.0f, z1 = 0.0f;
  int n1 = 0;
  auto fetch = [&](int e) {
    if (e < e_hi) {
      n1 = c.layer == 0 ? __ldg(a.xs_n + c.ebeg + e) : s0 + e;
      x1 = c.layer == 0 ? __ldg(a.xs_v + c.ebeg + e) : 0.0f;
      z1 = zrow[n1];
    }
  };
  const int e0 = q * a.SUB + (int)(threadIdx.x & 31);
  fetch(e0);
#pragma unroll 1
  for (int e = e0; e < e_hi; e += 32) {
    const int n = n1;
    float zn;
    const float da = entry_step<ACT1>(a, c, x1, z1, zn);
    fetch(e + 32);
    acc += vdelta<ACT2, LOSS, M, false>(a, R, onehot, dir, n - s0, da);
  }
  __syncwarp();
  return warp_sum(acc);
}

// Commit of a candidate that is not cached to this CTA's samples: thread i0 of istride.
template <int ACT1, int ACT2, int LOSS, int M>
__device__ __forceinline__ void commit_global(const Mlp2Args& a, const VRecs<M> R,
                                              const float* onehot, int s0, const Cand& c,
                                              const float* w2c, int i0, int istride) {
  float* zrow = a.z1 + (size_t)(c.layer == 0 ? c.row : c.col) * a.Np;
  const Direction<M> dir = direction<M>(c, w2c);
#pragma unroll 1
  for (int e = i0; e < c.ecnt; e += istride) {
    const int n = c.layer == 0 ? __ldg(a.xs_n + c.ebeg + e) : s0 + e;
    const float x = c.layer == 0 ? __ldg(a.xs_v + c.ebeg + e) : 0.0f;
    float zn;
    const float da = entry_step<ACT1>(a, c, x, zrow[n], zn);
    if (c.layer == 0) zrow[n] = zn;
    (void)vdelta<ACT2, LOSS, M, true>(a, R, onehot, dir, n - s0, da);
  }
}

// Warp prepares slot sl for trial t: proposal, W2 column, and (cacheable first-layer candidates)
// the gathered entries; then publishes it. `epoch` was read before any of the data.
template <int ACT1>
__device__ __forceinline__ void prepare_slot(const Mlp2Args& a, WSlot* slots, float (*w2c)[16],
                                             unsigned short* e_nl, float* e_da, float* e_zn,
                                             int sl, unsigned long long t, int epoch, int r, int s0,
                                             int s1) {
  const int lane = threadIdx.x & 31;
  if (lane == 0) {
    const uint4 w = trial_words(a.seed, t);
    const unsigned int idx = mlp2_trial_index(a.P, a.P1, a.seed, t, w.x, a.stretch);
    Cand c;
    fill_candidate(a, idx, w.y, false, 0.0f, r, s0, s1, c);
    slots[sl].c = c;
    slots[sl].epoch = epoch;
    slots[sl].theta = a.metro ? metropolis_theta_word(w.w, a.msc) : 0.0f;
  }
  __syncwarp();
  const Cand c = slots[sl].c;
  if (c.layer == 0 && c.gcnt > 0) {
    if (lane < 16) w2c[sl][lane] = lane < a.C ? a.w2[(size_t)lane * a.H + c.row] : 0.0f;
  }
  int state = 2;             // not cached: does not fit, or activation changes that are not finite
  bool finite = true;
  if (c.gcnt == 0) {
    state = 1;
  } else if (c.layer == 0 && c.ecnt <= kCap) {
    const float* zrow = a.z1 + (size_t)c.row * a.Np;
    unsigned short* nl = e_nl + (size_t)sl * kCap;
    float* da = e_da + (size_t)sl * kCap;
    float* zn = e_zn + (size_t)sl * kCap;
    for (int e0 = 0; e0 < c.ecnt; e0 += 128) {
      int nn[4];
      float xv[4], zv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * 32 + lane;
        nn[u] = -1;
        xv[u] = 0.0f;
        if (e < c.ecnt) {
          nn[u] = __ldg(a.xs_n + c.ebeg + e);
          xv[u] = __ldg(a.xs_v + c.ebeg + e);
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) zv[u] = nn[u] >= 0 ? zrow[nn[u]] : 0.0f;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * 32 + lane;
        if (nn[u] < 0) continue;
        const float z2 = fmaf(c.delta, xv[u], zv[u]);
        nl[e] = (unsigned short)(nn[u] - s0);
        zn[e] = z2;
        const float d = act_compact<ACT1>(z2, a.g1, a.act1) - act_compact<ACT1>(zv[u], a.g1, a.act1);
        da[e] = d;
        finite &= fabsf(d) < INFINITY;
      }
    }
    state = __all_sync(0xffffffffu, finite) ? 1 : 2;
  }
  __syncwarp();
  if (lane == 0) {
    slots[sl].state = state;
    st_release_cta_shared_u64(&slots[sl].ticket, t + 1ull);
  }
  __syncwarp();
}

// Acquires the data of trial t's slot when it is ready.
__device__ __forceinline__ bool slot_ready(const WSlot& s, unsigned long long t) {
  return ld_acquire_cta_shared_u64(&s.ticket) == t + 1ull;
}

// Slot k places after slot sl (both below kWS).
__device__ __forceinline__ int slot_after(int sl, int k) {
  const int v = sl + k;
  return v >= kWS ? v - kWS : v;
}

// The warp replays the commits [slot epoch, epoch) on a ready slot, 32 log entries at a time.
// Returns false (in every lane) when the slot must be prepared again.
__device__ __forceinline__ bool revalidate(WSlot& s, float* w2c, const CommitLog* log, int epoch) {
  const int lane = threadIdx.x & 31;
  const int e0 = s.epoch;
  if (epoch - e0 >= kLogLen) return false;
  const unsigned int idx = s.c.idx;
  const int layer = s.c.layer, row = s.c.row;
  for (int base = e0; base < epoch; base += 32) {
    const int e = base + lane;
    bool stale = false, patch = false;
    int prow = 0;
    float pval = 0.0f;
    if (e < epoch) {
      const CommitLog& L = log[e % kLogLen];
      stale = L.idx == idx || (layer == 0 && L.layer == 0 && L.changes_z1 && L.row == row);
      patch = layer == 0 && L.layer == 1 && L.col == row;
      prow = L.row;
      pval = L.neww;
    }
    if (__any_sync(0xffffffffu, stale)) return false;
    unsigned int pm = __ballot_sync(0xffffffffu, patch);
    while (pm) {                       // in commit order: the latest value of a row wins
      const int j = __ffs(pm) - 1;
      pm &= pm - 1u;
      if (lane == j) w2c[prow] = pval;
      __syncwarp();
    }
  }
  __syncwarp();
  if (lane == 0) s.epoch = epoch;
  __syncwarp();
  return true;
}

// One lane brings a ready slot from epoch E - 1 to E with log entry L (commit E - 1). Returns false
// when the slot must be prepared again.
__device__ __forceinline__ bool replay_one(WSlot& o, float* w2c, const CommitLog& L, int E) {
  const Cand& c = o.c;
  if (L.idx == c.idx || (c.layer == 0 && L.layer == 0 && L.changes_z1 && L.row == c.row))
    return false;
  if (c.layer == 0 && L.layer == 1 && L.col == c.row) w2c[L.row] = L.neww;
  o.epoch = E;
  return true;
}

// What a warp knows about 32 slots, one bit per lane: ready and up to date, a valid proposal, a live
// one (something to evaluate).
struct SlotBits {
  unsigned int ready, valid, live;
};

__device__ __forceinline__ SlotBits slot_bits(const WSlot& o, bool ready) {
  bool valid = false, live = false;
  if (ready) {
    valid = o.c.valid != 0;
    live = valid && o.c.gcnt > 0;
  }
  SlotBits b;
  b.ready = __ballot_sync(0xffffffffu, ready);
  b.valid = __ballot_sync(0xffffffffu, valid);
  b.live = __ballot_sync(0xffffffffu, live);
  return b;
}

// Bits [at, at + 64) of three words (bits past the 96th are 0); 0 <= at <= 64.
__device__ __forceinline__ unsigned long long window_bits(const unsigned int* w, int at) {
  const unsigned long long lo = (unsigned long long)w[1] << 32 | w[0], hi = w[2];
  if (at == 0) return lo;
  if (at == 64) return hi;
  return lo >> at | hi << (64 - at);
}

// This range's loss change of a candidate, added into the candidate's packed 64-bit word: bits
// 56..63 count the CTAs that have added, bits 48..55 those whose share was not finite or not below
// 2^19 in magnitude, bits 0..47 the sum over the CTAs of (share in units of 2^-20) + 2^39. Integer sums
// are exact and independent of the order of arrival, so dS is the same in every CTA and for every
// batch width; the count is the batch's only grid-wide wait, and one load of the word gives
// everything.
__device__ __forceinline__ void add_share(unsigned long long* word, float sum) {
  unsigned long long w = 1ull << 56;
  if (isfinite(sum) && fabsf(sum) < 0x1p19f)
    w += (1ull << 39) + (unsigned long long)__float2ll_rn(sum * 0x1p20f);
  else
    w += 1ull << 48;
  atomicAdd(word, w);
}

// Compulsory bytes of the batch's candidates not evaluated before (statistics of CTA 0).
__device__ __forceinline__ unsigned long long batch_bytes(const WSlot* slots, unsigned long long tau,
                                                          int Kb, int sl_tau,
                                                          unsigned long long tau_hi) {
  const int lane = threadIdx.x & 31;
  unsigned long long bytes = 0ull;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int k = lane + 32 * h;
    if (k < Kb && tau + (unsigned long long)k >= tau_hi)
      bytes += slots[slot_after(sl_tau, k)].c.bytes;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) bytes += __shfl_xor_sync(0xffffffffu, bytes, o);
  return bytes;
}

// M: fields of a sample's record (10 for up to 10 classes, else 14).
template <int ACT1, int ACT2, int LOSS, int M>
__global__ void __launch_bounds__(kLoopThreads, 1) mlp2_window_loop(Mlp2Args a) {
  extern __shared__ __align__(16) float s_dyn[];
  __shared__ WSlot s_slot[kWS];
  __shared__ __align__(16) float s_w2c[kWS][16];
  __shared__ __align__(16) float s_onehot[16][16];   // -[k == y]
  __shared__ float s_sub[kWinBatch][kMaxSubs];        // sums of a candidate's chunks
  __shared__ CommitLog s_log[kLogLen];
  __shared__ float s_dS[kWinBatch];
  __shared__ unsigned int s_stale[2];
  // the slots kWS places on from the batch's first trial, as the last look found them: words of 32
  // slots, [0] ready and up to date, [1] valid, [2] live
  __shared__ unsigned int s_bits[3][kWS / 32];
  __shared__ unsigned long long s_live;               // the batch's live candidates, if not as found
  __shared__ int s_flag, s_kstar, s_bvalid, s_fail, s_done, s_epoch, s_redo;
  __shared__ int s_cnt[kWinBatch];     // warps done with a candidate
  // trials whose slots a commit made stale ahead of their batch, for the producers to prepare
  // again: entry (position mod kRedoLen) holds trial + 1 once written, 0 once taken
  __shared__ unsigned long long s_redo_q[kRedoLen];
  __shared__ unsigned int s_redo_head, s_redo_tail;
  __shared__ unsigned long long s_bbytes, s_tau_hi, s_next, s_limit;
  // CTA 0's statistics, here rather than in 20 registers of every thread: with them the kernels spill, and a
  // batch of the wide net took 4.07 us instead of 3.89
  __shared__ unsigned long long s_cand, s_waste, s_bytes, s_bytes_back, s_trace;
  __shared__ double s_S;
  float* s_records = s_dyn;
  unsigned short* e_nl = reinterpret_cast<unsigned short*>(s_dyn + kRecFields * a.RS);
  float* e_da = reinterpret_cast<float*>(e_nl + kWS * kCap);
  float* e_zn = e_da + kWS * kCap;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r = blockIdx.x;
  const int s0 = min(r * a.RS, a.N), s1 = min(s0 + a.RS, a.N);
  const VRecs<M> R{s_records};
  const float* onehot = &s_onehot[0][0];
  {
    // the records: fields past the class count hold -infinity
    const int ns = s1 - s0;
#pragma unroll 1
    for (int f = 0; f < M + 2; ++f)
#pragma unroll 1
      for (int nl = tid; nl < ns; nl += kLoopThreads)
        R.at(nl, f) = f < M && f >= a.C
                          ? -INFINITY
                          : a.srec[(size_t)(f < M ? f : f - M + kRecLoss) * a.Np + s0 + nl];
    for (int q = tid; q < 256; q += kLoopThreads)
      s_onehot[q >> 4][q & 15] = (q >> 4) == (q & 15) ? -1.0f : 0.0f;
  }
  for (int q = tid; q < kWS; q += kLoopThreads) s_slot[q].ticket = 0ull;
  for (int q = tid; q < kRedoLen; q += kLoopThreads) s_redo_q[q] = 0ull;
  for (int q = tid; q < kWinBatch; q += kLoopThreads) s_cnt[q] = 0;
  DevState* st = a.st;
  unsigned long long tau = a.tau0;
  const unsigned long long end = a.tau0 + a.n_trials;
  if (tid == 0) {
    s_tau_hi = a.tau0;
    s_cand = s_waste = s_bytes = s_bytes_back = 0ull;
    s_trace = st->trace_written;
    s_S = st->S;
    s_next = a.tau0;
    s_limit = a.tau0 + (unsigned long long)window_lead(a.H, 1);
    s_redo_head = s_redo_tail = 0u;
    s_fail = 0;
    s_done = 0;
    s_epoch = 0;
    for (int q = 0; q < kWS / 32; ++q) s_bits[0][q] = 0u;
  }
  __syncthreads();

  if (warp >= kConsWarps) {
    // ---- producers: slots to prepare again first, then new ones in trial order up to s_limit
    unsigned long long tn = 0ull;      // lane 0: the next new trial this warp took
    bool have = false;
    unsigned int n_again = 0;
    for (;;) {
      unsigned long long t = ~0ull;
      if (lane == 0) {
        unsigned long long w0 = 0ull;
        unsigned int spins = 0;
        for (;;) {
          const unsigned int tl = *(volatile unsigned int*)&s_redo_tail;
          // 0: no entry, or its writer is between two stores (looked at again after a new trial, or in the
          // bounded wait below)
          const unsigned long long e = ld_acquire_cta_shared_u64(&s_redo_q[tl % kRedoLen]);
          if (e != 0ull) {
            if (atomicCAS(&s_redo_tail, tl, tl + 1u) == tl) {
              t = e - 1ull;
              st_release_cta_shared_u64(&s_redo_q[tl % kRedoLen], 0ull);
              ++n_again;
              break;
            }
            continue;                  // another producer took it
          }
          if (!have) {
            tn = atomicAdd(&s_next, 1ull);
            have = true;
          }
          if (tn < end && tn < *(volatile unsigned long long*)&s_limit) {
            t = tn;
            have = false;
            break;
          }
          if (*(volatile int*)&s_done) break;
          if ((++spins & 63u) == 0u) {
            const unsigned long long now = globaltimer_ns();
            if (w0 == 0ull) {
              w0 = now;
            } else if (now - w0 > kBarrierTimeoutNs) {
              atomicCAS(&st->err, 0, (int)MCA_ERR_TIMEOUT);   // the consumers stop at their decision
              break;
            }
          }
          __nanosleep(64);
        }
      }
      t = __shfl_sync(0xffffffffu, t, 0);
      if (t == ~0ull) break;
      int epoch = 0;
      if (lane == 0) epoch = ld_acquire_cta_shared_s32(&s_epoch);
      __syncwarp();
      epoch = __shfl_sync(0xffffffffu, epoch, 0);
      prepare_slot<ACT1>(a, s_slot, s_w2c, e_nl, e_da, e_zn, (int)(t % kWS), t, epoch, r, s0, s1);
    }
    if (lane == 0 && n_again) atomicAdd(&st->phase_ns[7], (unsigned long long)n_again);
  } else {
    // ---- consumers: the batches. The commit of batch b runs at the start of batch b + 1 on warps
    // 1.., overlapped with that batch's set-up on warp 0, which reads neither records nor z1.
    const bool stats_thread = r == 0 && tid == 0;
    const bool timer = kPhaseTimers && tid == 0;   // phase times of every CTA, mean over CTAs
    unsigned long long ph0 = 0, ph1 = 0, ph2 = 0, ph3 = 0, n_starve = 0;
    unsigned int n_reprep = 0;
    float rate_a = st->rate_acc, rate_t = st->rate_trials;
    unsigned int bidx = 0;
    int epoch = 0;                     // commits of this CTA so far (consumer copy of s_epoch)
    const int kmaxw = min(a.K, kWinBatch);
    int sl_tau = (int)(tau % kWS);     // slot of trial tau
    int pend = -1;                     // slot of the accepted candidate not yet committed
    int adv = 0;                       // trials the previous batch consumed
    int kst = -1;                      // its accepted candidate
    CommitLog mine[2];                 // warp 0: the log entries of this lane's candidates if accepted
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      mine[h].idx = ~0u;
      mine[h].layer = mine[h].row = mine[h].col = -1;
      mine[h].neww = 0.0f;
      mine[h].changes_z1 = 0;
    }
    int nlive = 0, wpc = 1;            // live candidates of the batch, warps per candidate
    bool held = false;                 // each of them had its own warps, warp 0 none
    int hk = -1, he = 0;               // the candidate of this warp's last chunk of cached entries, the
    float hl = 0.0f;                   // lane's entry, and its new loss

    for (;;) {
      const unsigned long long t_a = timer ? globaltimer_ns() : 0ull;
      const bool more = tau < end;
      int Kb = 0;
      if (more) {
        const int Kw = a.fixed_K ? kmaxw : batch_width_fast(rate_a, rate_t, a.wscale, kmaxw);
        Kb = (int)((end - tau) < (unsigned long long)Kw ? (end - tau) : Kw);
      }
      const int E = epoch + (pend >= 0 ? 1 : 0);    // commits including the pending one
      // every warp: are the batch's slots all ready, and which are live, by the last look
      const unsigned long long want = Kb >= 64 ? ~0ull : (1ull << Kb) - 1ull;
      const bool known = (window_bits(s_bits[0], adv) & want) == want;
      const unsigned long long valid_mask = window_bits(s_bits[1], adv) & want;
      unsigned long long live_mask = window_bits(s_bits[2], adv) & want;
      if (warp == 0) {
        // ---- set-up: every slot of the batch ready and brought up to E, lane k (and k + 32) for
        // batch position k. Usually the previous batch's look found them all ready and at `epoch`,
        // and only the pending commit (P) has to be checked against them; otherwise a bounded wait
        // for the producers and a replay of the log.
        const int nh = Kb > 32 ? 2 : 1;
        CommitLog P;                   // the pending commit's log entry (pend >= 0: kst >= 0)
        P.idx = ~0u;
        P.layer = P.row = P.col = -1;
        P.neww = 0.0f;
        P.changes_z1 = 0;
        if (kst >= 0) {                // the accepted candidate's log entry, from its lane
          const bool up = kst >= 32;
          const int j = kst & 31;
          P.idx = __shfl_sync(0xffffffffu, up ? mine[1].idx : mine[0].idx, j);
          P.layer = __shfl_sync(0xffffffffu, up ? mine[1].layer : mine[0].layer, j);
          P.row = __shfl_sync(0xffffffffu, up ? mine[1].row : mine[0].row, j);
          P.col = __shfl_sync(0xffffffffu, up ? mine[1].col : mine[0].col, j);
          P.neww = __shfl_sync(0xffffffffu, up ? mine[1].neww : mine[0].neww, j);
          P.changes_z1 =
              __shfl_sync(0xffffffffu, up ? mine[1].changes_z1 : mine[0].changes_z1, j);
        }
        if (lane == 0)     // producers may fill slots up to the limit past the oldest in use
          *(volatile unsigned long long*)&s_limit =
              (pend >= 0 ? tau - 1ull : tau) + (unsigned long long)window_lead(a.H, Kb);
        bool full[2] = {false, false}, stale[2] = {false, false};
        unsigned int mf0 = 0u, mf1 = 0u;
        int sl[2];
        sl[0] = slot_after(sl_tau, min(lane, max(Kb - 1, 0)));
        sl[1] = slot_after(sl_tau, min(lane + 32, max(Kb - 1, 0)));
        if (known) {
          if (pend >= 0) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              if (h >= nh) break;
              if (lane + 32 * h < Kb)
                stale[h] = !replay_one(s_slot[sl[h]], s_w2c[sl[h]], P, E);
            }
          }
          if (pend >= 0 && lane == 0) s_log[epoch % kLogLen] = P;
        } else {
          SlotBits b[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int k = lane + 32 * h;
            bool ok = k < Kb;
            WSlot& o = s_slot[sl[h]];
            if (ok) {
              const unsigned long long t = tau + (unsigned long long)k;
              unsigned long long w0 = kPhaseTimers ? globaltimer_ns() : 0ull;
              unsigned int spins = 0;
              while (!slot_ready(o, t)) {
                if ((++spins & 63u) == 0u) {
                  const unsigned long long now = globaltimer_ns();
                  if (w0 == 0ull) {
                    w0 = now;
                  } else if (now - w0 > kBarrierTimeoutNs) {
                    atomicCAS(&st->err, 0, (int)MCA_ERR_TIMEOUT);
                    *(volatile int*)&s_fail = 1;
                    ok = false;
                    break;
                  }
                }
              }
              if (kPhaseTimers) n_starve += globaltimer_ns() - w0;
            }
            if (ok) {
              const int oe = o.epoch;
              if (oe == E - 1 && pend >= 0)
                stale[h] = !replay_one(o, s_w2c[sl[h]], P, E);
              else if (oe != E)
                full[h] = true;
            }
            __syncwarp();
            b[h] = slot_bits(o, ok);
          }
          if (lane == 0) {
            s_live = (unsigned long long)b[1].live << 32 | b[0].live;
            s_bvalid = __popc(b[0].valid) + __popc(b[1].valid);
            if (pend >= 0) s_log[epoch % kLogLen] = P;
          }
          mf0 = __ballot_sync(0xffffffffu, full[0]);
          mf1 = __ballot_sync(0xffffffffu, full[1]);
        }
        if (mf0 | mf1) {
          // older commits to replay (slots published after the last look): warp-wide, rare
          __syncwarp();
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            unsigned int m = h ? mf1 : mf0;
            while (m) {
              const int j = __ffs(m) - 1;
              m &= m - 1u;
              const int slj = __shfl_sync(0xffffffffu, sl[h], j);
              const bool okj = revalidate(s_slot[slj], s_w2c[slj], s_log, E);
              if (lane == j) stale[h] = !okj;
            }
          }
        }
        const unsigned int ms0 = __ballot_sync(0xffffffffu, stale[0]);
        const unsigned int ms1 = __ballot_sync(0xffffffffu, stale[1]);
        if (lane == 0) {
          s_stale[0] = ms0;
          s_stale[1] = ms1;
          s_redo = (ms0 | ms1) != 0u || *(volatile int*)&s_fail != 0;
        }
      } else if (pend >= 0) {
        // ---- commit of the pending candidate to this CTA's samples (threads 32..)
        const int sl = pend;
        const Cand c = s_slot[sl].c;
        const int i0 = tid - 32, istride = kConsThreads - 32;
        if (c.gcnt > 0) {
          if (s_slot[sl].state == 1) {
            float* zrow = a.z1 + (size_t)c.row * a.Np + s0;
            const unsigned short* nl = e_nl + (size_t)sl * kCap;
            const float* da = e_da + (size_t)sl * kCap;
            const float* zn = e_zn + (size_t)sl * kCap;
            float2 w[M / 2];
            load_column<M>(s_w2c[sl], w);
            if (held && (c.ecnt + 31) / 32 <= wpc) {
              // every entry was the last one of some lane of warps 1.., which has its new loss: the
              // losses are not computed again (a batch of the wide net 4.28 us with, 4.06 without
              // computing them; keeping the fields as well spills registers)
              if (hk == kst && he < c.ecnt) commit_entry<M>(R, w, nl, da, zn, he, hl, zrow);
            } else {
#pragma unroll 1
              for (int e = i0; e < c.ecnt; e += istride) {
                float2 z[M / 2];
                float ln;
                int n, y;
                (void)cached_entry<ACT2, LOSS, M>(a, R, onehot, w, s_w2c[sl], nl, da, e, c.ecnt, z,
                                                  ln, n, y);
                zrow[n] = zn[e];
                if (da[e] != 0.0f) R.store(n, z, ln, y);
              }
            }
          } else {
            commit_global<ACT1, ACT2, LOSS, M>(a, R, onehot, s0, c, s_w2c[sl], i0, istride);
          }
        }
        if (tid == 32) {
          if (r == 0 && c.layer == 0 && c.gcnt > 0)   // hidden-field sectors written back
            s_bytes_back += 32ull * (unsigned long long)a.xs_sect[c.col];
          const unsigned long long off = c.idx - (c.layer ? a.P1 : 0ull);
          (c.layer ? a.w2 : a.w1)[off] = c.neww;
          const int wk = c.layer ? a.wk2 : a.wk1;
          if (wk != MCA_W_FP32) (c.layer ? a.code2 : a.code1)[off] = (signed char)c.new_code;
        }
      }
      // this warp's part of the evaluation (below), ahead of the barrier where the live candidates are
      // known; warp 0, which ends the set-up, after it
      int vi = 0, vj = 0, vk = 0;
      auto split = [&]() {
        const int vw = warp == 0 ? kConsWarps - 1 : warp - 1;
        nlive = __popcll(live_mask);
        const int x = min(max(nlive, 1) - 1, kWpcLast);
        wpc = (int)(kWpc >> (4 * x)) & 15;
        vi = (vw * ((int)(kWpcInv >> (9 * x)) & 511)) >> 8;
        vj = vw - vi * wpc;
        vk = nth_bit(live_mask, vi);
      };
      if (known && warp != 0) split();
      cons_sync();
      if (pend >= 0) {
        // every consumer's writes of the commit precede the new epoch that producers read
        ++epoch;
        if (tid == 0) st_release_cta_shared_s32(&s_epoch, epoch);
        pend = -1;
      }
      if (!more) break;
      const bool redo = s_redo != 0;
      if (redo) {
        if (*(volatile int*)&s_fail) break;
        // slots the commit invalidated, prepared again now that it is complete, one per warp
        int turn = 0;
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          unsigned int m = s_stale[h];
          while (m) {
            const int j = __ffs(m) - 1;
            m &= m - 1u;
            if (turn == warp) {
              const int k = j + 32 * h;
              prepare_slot<ACT1>(a, s_slot, s_w2c, e_nl, e_da, e_zn, slot_after(sl_tau, k),
                                 tau + (unsigned long long)k, epoch, r, s0, s1);
              if (lane == 0) ++n_reprep;
            }
            turn = turn + 1 == kConsWarps ? 0 : turn + 1;
          }
        }
        cons_sync();
        if (warp == 0) {               // a slot's candidate may have become live, or dead
          SlotBits b[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int k = lane + 32 * h;
            b[h] = slot_bits(s_slot[slot_after(sl_tau, min(k, Kb - 1))], k < Kb);
          }
          if (lane == 0) {
            s_live = (unsigned long long)b[1].live << 32 | b[0].live;
            s_bvalid = __popc(b[0].valid) + __popc(b[1].valid);
          }
        }
        cons_sync();
      }
      const unsigned long long t_s = timer ? globaltimer_ns() : 0ull;
      if (!known || redo) live_mask = s_live;
      if (!known || redo || warp == 0) split();
      held = nlive < kConsWarps;
      hk = -1;
      // ---- evaluate. A candidate's entries in this range are cut into chunks: 32 cached entries (from
      // shared memory), or a.SUB samples read from global memory. What bounds the evaluation is the
      // length of one warp's instruction sequence, so the warps share the candidates: wpc warps per
      // candidate, warp j of them taking chunks j, j + wpc, ... (a batch of 4096 Gaussian neurons,
      // 80 entries a candidate: 4.24 us with one warp per candidate, 3.79 with two to four). The chunks
      // are fixed by the candidate and added in order, whatever the number of warps. The warp that
      // finishes a candidate adds the CTA's share. The last three warps look at the slots ahead: before
      // they evaluate when the others suffice for that, else afterwards. Warp 0, which waits for the
      // other CTAs, is the last to get work. Each warp's part comes from tables, ahead of the
      // barrier: with three divisions after it a batch of the wide net took 4.40 us, with the tables
      // 4.28.
      unsigned long long* acc = a.accum + (size_t)(bidx % kAccBuffers) * kAccStride;
      const bool look_first = nlive * wpc <= kLookWarp0 - 1;
#pragma unroll 1
      for (int ph = 0; ph < 2; ++ph) {
        if ((ph == 0) == look_first) {
          if (warp < kLookWarp0) continue;
          // the published slots up to kWS trials on, brought up to `epoch`, one slot per lane (a few
          // commits behind: replayed by the lane; further: warp-wide); a stale slot goes back to the
          // producers and is not ready until they are done
          const int j = lane + 32 * (warp - kLookWarp0);
          const unsigned long long t = tau + (unsigned long long)j;
          const int slj = slot_after(sl_tau, j);
          WSlot& o = s_slot[slj];
          bool ready = t < end && slot_ready(o, t), full = false, again = false;
          if (ready && j >= Kb) {
            const int lag = epoch - o.epoch;
            if (lag > 4) {
              full = true;
            } else {
              for (int e = o.epoch; e < epoch; ++e)
                if (!replay_one(o, s_w2c[slj], s_log[e % kLogLen], e + 1)) {
                  again = true;
                  break;
                }
            }
          }
          unsigned int m = __ballot_sync(0xffffffffu, full);
          while (m) {
            const int jj = __ffs(m) - 1;
            m &= m - 1u;
            const int sj = __shfl_sync(0xffffffffu, slj, jj);
            const bool ok = revalidate(s_slot[sj], s_w2c[sj], s_log, epoch);
            if (lane == jj) again = !ok;
          }
          if (again) {
            ready = false;
            o.ticket = 0ull;
            const unsigned int p = atomicAdd(&s_redo_head, 1u);
            st_release_cta_shared_u64(&s_redo_q[p % kRedoLen], t + 1ull);
          }
          const SlotBits b = slot_bits(o, ready);
          if (lane == 0) {
            s_bits[0][warp - kLookWarp0] = b.ready;
            s_bits[1][warp - kLookWarp0] = b.valid;
            s_bits[2][warp - kLookWarp0] = b.live;
          }
          continue;
        }
#pragma unroll 1
        for (int i = vi; i < nlive; i += kConsWarps) {         // (wpc = 1 when there are more)
          const int j = vj, k = i == vi ? vk : nth_bit(live_mask, i);
          const int sl = slot_after(sl_tau, k);
          const Cand& c = s_slot[sl].c;
          const bool cached = s_slot[sl].state == 1;
          const int nc = max(1, cached ? (c.ecnt + 31) / 32 : c.nsub);
          if (j >= nc) break;              // fewer chunks than warps
          const bool alone = wpc == 1 || nc == 1;
          float v = 0.0f;
          if (cached) {
            float2 w[M / 2];
            load_column<M>(s_w2c[sl], w);
            hk = k;
#pragma unroll 1
            for (int q = j; q < nc; q += wpc) {
              float2 z[M / 2];
              int n, y;
              he = 32 * q + lane;
              const float t = warp_sum(cached_entry<ACT2, LOSS, M>(
                  a, R, onehot, w, s_w2c[sl], e_nl + (size_t)sl * kCap, e_da + (size_t)sl * kCap, he,
                  c.ecnt, z, hl, n, y));
              v += t;
              if (!alone && lane == 0) s_sub[k][q] = t;
            }
          } else {
#pragma unroll 1
            for (int q = j; q < nc; q += wpc) {
              const float t = eval_global<ACT1, ACT2, LOSS, M>(a, R, onehot, s0, c, s_w2c[sl], q);
              v += t;
              if (!alone && lane == 0) s_sub[k][q] = t;
            }
          }
          if (lane == 0) {
            bool last = true;
            if (!alone) {
              __threadfence_block();
              last = atomicAdd(&s_cnt[k], 1) == min(wpc, nc) - 1;
              if (last) {
                __threadfence_block();
                s_cnt[k] = 0;
                v = 0.0f;
                for (int u = 0; u < nc; ++u) v += *(volatile float*)&s_sub[k][u];
              }
            }
            if (last) add_share(acc + k * kAccWord, v);
          }
          __syncwarp();
        }
      }
      // CTA 0 clears the buffer of batch bidx + 2, which is also that of batch bidx - 2: every CTA
      // has added its share of batch bidx - 1, so every CTA has finished waiting on batch
      // bidx - 2. The clearing is fenced before the barrier that ends this batch in CTA 0, so before
      // its additions to batch bidx + 1, for which every CTA waits before it adds to batch bidx + 2.
      if (r == 0 && warp == kLookWarp0 - 1) {
        unsigned long long* z = a.accum + (size_t)((bidx + 2) % kAccBuffers) * kAccStride;
        z[lane * kAccWord] = 0ull;
        z[(lane + 32) * kAccWord] = 0ull;
        if (lane == 0) z[kArrivalWord * kAccWord] = 0ull;
        __threadfence();
      }
      // a batch without a live candidate still synchronises (on the arrival word), so that no
      // CTA runs more than one batch ahead of the clearing of the rotating buffers
      if (tid == 0 && live_mask == 0ull) atomicAdd(acc + kArrivalWord * kAccWord, 1ull << 56);
      const unsigned long long t_b = timer ? globaltimer_ns() : 0ull;
      const int nvalid = known && !redo ? __popcll(valid_mask) : s_bvalid;
      // ---- warp 0 waits until every CTA has added to every live candidate (bounded), then
      // decides
      if (warp == 0) {
        const unsigned long long need = (unsigned long long)gridDim.x;
        int ok = 1;
        unsigned long long v[2] = {0ull, 0ull};
        const int nh = Kb > 32 ? 2 : 1;
        bool live[2] = {false, false}, valid[2] = {false, false}, poll[2];
        float theta[2] = {0.0f, 0.0f};
        const unsigned long long* pa[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k = lane + 32 * h;
          mine[h].idx = ~0u;
          mine[h].layer = mine[h].row = mine[h].col = -1;
          mine[h].neww = 0.0f;
          mine[h].changes_z1 = 0;
          if (h < nh && k < Kb) {
            const WSlot& o = s_slot[slot_after(sl_tau, k)];
            valid[h] = o.c.valid != 0;
            live[h] = valid[h] && o.c.gcnt > 0;
            theta[h] = o.theta;
            mine[h].idx = o.c.idx;
            mine[h].layer = o.c.layer;
            mine[h].row = o.c.row;
            mine[h].col = o.c.col;
            mine[h].neww = o.c.neww;
            mine[h].changes_z1 = o.c.layer == 0 && o.c.gcnt > 0;
          }
          poll[h] = live[h];
          pa[h] = acc + k * kAccWord;
        }
        if (live_mask == 0ull && lane == 0) {
          poll[0] = true;
          pa[0] = acc + kArrivalWord * kAccWord;
        }
        // the clock is read only once the wait has lasted 64 polls (and for the phase timers)
        unsigned long long w0 = kPhaseTimers ? globaltimer_ns() : 0ull;
        unsigned int spins = 0;
        for (;;) {
          bool mine = true;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (poll[h] && (v[h] >> 56) < need) {
              v[h] = ld_acquire_gpu_u64(pa[h]);
              mine = mine && (v[h] >> 56) >= need;
            }
          }
          if (__all_sync(0xffffffffu, mine)) break;
          int stop = 0;
          if (lane == 0 && (++spins & 63u) == 0u) {
            const unsigned long long now = globaltimer_ns();
            if (spins == 64u && !kPhaseTimers) w0 = now;
            if (ld_volatile_int(&st->err) != 0) {
              stop = 1;
            } else if (now - w0 > kBarrierTimeoutNs) {
              atomicCAS(&st->err, 0, (int)MCA_ERR_TIMEOUT);
              stop = 1;
            }
          }
          if (__shfl_sync(0xffffffffu, stop, 0)) {
            ok = 0;
            break;
          }
        }
        // decide in the same warp (the same in every CTA): lowest-index candidate with
        // dS <= theta (Eq. 6 / Eq. 7); decisions forced by the caller take precedence; a
        // non-finite dS at or before the first acceptance stops the run
        unsigned int mask_a[2] = {0u, 0u}, mask_b[2] = {0u, 0u}, mask_f[2] = {0u, 0u};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (h >= nh) break;
          const int k = lane + 32 * h;
          bool accept = false, bad = false, forced = false;
          if (k < Kb) {
            float d = 0.0f;
            const unsigned long long nbad = (v[h] >> 48) & 255ull;
            if (!valid[h] || (live[h] && nbad != 0ull)) {
              d = __int_as_float(0x7fc00000);
            } else if (live[h]) {
              const long long q =
                  (long long)(v[h] & ((1ull << 48) - 1ull)) - (long long)(need << 39);
              d = __ll2float_rn(q) * 0x1p-20f;
            }
            s_dS[k] = d;
            if (valid[h]) {
              const unsigned long long tk = tau + (unsigned long long)k;
              bool facc = false;
              if (a.nforce > 0) {
                int lo = 0, hi = a.nforce;
                while (lo < hi) {
                  const int mid = (lo + hi) >> 1;
                  if (a.ftau[mid] < tk)
                    lo = mid + 1;
                  else
                    hi = mid;
                }
                if (lo < a.nforce && a.ftau[lo] == tk) {
                  forced = true;
                  facc = a.facc[lo] != 0;
                }
              }
              if (forced) {
                accept = facc;
              } else {
                bad = !isfinite(d);
                accept = a.strict ? d < theta[h] : d <= theta[h];
              }
            }
          }
          mask_a[h] = __ballot_sync(0xffffffffu, accept);
          mask_b[h] = __ballot_sync(0xffffffffu, bad);
          mask_f[h] = __ballot_sync(0xffffffffu, forced);
        }
        __syncwarp();
        int kstar = mask_a[0] ? __ffs(mask_a[0]) - 1 : (mask_a[1] ? 31 + __ffs(mask_a[1]) : -1);
        const int kbad =
            mask_b[0] ? __ffs(mask_b[0]) - 1 : (mask_b[1] ? 31 + __ffs(mask_b[1]) : -1);
        if (kbad >= 0 && (kstar < 0 || kbad <= kstar)) kstar = -2;
        if (lane == 0) {
          if (kPhaseTimers) ph2 += globaltimer_ns() - w0;
          s_flag = ok;                 // an error elsewhere ends this CTA's next wait
          s_kstar = kstar;
          if (stats_thread && ok) {
            const int last = kstar >= 0 ? kstar : Kb - 1;
            if (a.trace_cap > 0) {
              for (int k = 0; k <= last; ++k) {
                const Cand& c = s_slot[slot_after(sl_tau, k)].c;
                mca_trace_rec rec;
                rec.tau = tau + (unsigned long long)k;
                rec.idx = c.idx;
                rec.accept = k == kstar ? 1 : 0;
                rec.old_w = c.oldw;
                rec.new_w = c.neww;
                rec.valid = c.valid;
                rec.forced = (int)((mask_f[k >> 5] >> (k & 31)) & 1u);
                rec.dS = (double)s_dS[k];
                rec.S = s_S;
                a.trace[s_trace % (unsigned long long)a.trace_cap] = rec;
                ++s_trace;
              }
            }
#pragma unroll
            for (int w = 0; w < 2; ++w) {
              unsigned int m = mask_f[w];
              const int hi = last - w * 32;
              if (hi < 31) m &= hi < 0 ? 0u : ((2u << hi) - 1u);
              if (m) atomicAdd(&st->forced, (unsigned long long)__popc(m));
            }
            s_cand += (unsigned long long)nvalid;
            if (kstar >= 0) {
              s_waste += (unsigned long long)(Kb - kstar - 1);
              s_S += (double)s_dS[kstar];
            }
          }
        }
      } else if (warp == 1 && r == 0) {
        const unsigned long long bb = batch_bytes(s_slot, tau, Kb, sl_tau, s_tau_hi);
        if (lane == 0) s_bbytes = bb;
      }
      cons_sync();
      if (!s_flag) break;
      const int kstar = s_kstar;
      if (stats_thread) s_bytes += s_bbytes;
      if (timer) {
        const unsigned long long t_c = globaltimer_ns();
        ph0 += t_s - t_a;
        ph1 += t_b - t_s;
        ph3 += t_c - t_b;
      }
      if (kstar == -2) {
        if (stats_thread) {
          atomicCAS(&st->err, 0, (int)MCA_ERR_NUMERIC);
          st->batches += 1ull;         // (the others are counted below)
        }
        break;
      }
      if (tid == 0) s_tau_hi = max(s_tau_hi, tau + (unsigned long long)Kb);
      adv = kstar >= 0 ? kstar + 1 : Kb;
      kst = kstar;
      if (kstar >= 0) {
        pend = slot_after(sl_tau, kstar);
        rate_a = rate_a * kRateDecay + 1.0f;
      } else {
        rate_a = rate_a * kRateDecay;
      }
      rate_t = rate_t * kRateDecay + (float)adv;
      tau += (unsigned long long)adv;
      sl_tau = slot_after(sl_tau, adv);
      ++bidx;
    }
    if (tid == 0) *(volatile int*)&s_done = 1;
    if (timer) {
      const unsigned long long g = (unsigned long long)gridDim.x;
      atomicAdd(&st->phase_ns[0], ph0 / g);
      atomicAdd(&st->phase_ns[1], ph1 / g);
      atomicAdd(&st->phase_ns[2], ph2 / g);
      atomicAdd(&st->phase_ns[3], ph3 / g);
    }
    if (lane == 0 && (n_starve || n_reprep)) {
      atomicAdd(&st->phase_ns[6], n_starve / (unsigned long long)gridDim.x);
      atomicAdd(&st->phase_ns[7], (unsigned long long)n_reprep);
    }
    if (r == 0 && tid == 32 && s_bytes_back) atomicAdd(&st->alg_bytes, s_bytes_back);
    if (stats_thread) {
      st->S = s_S;
      st->trials += tau - a.tau0;
      st->accepts += (unsigned long long)epoch;        // every commit of this launch
      st->candidates += s_cand;
      st->batches += (unsigned long long)bidx;
      st->wasted += s_waste;
      atomicAdd(&st->alg_bytes, s_bytes);
      st->trace_written = s_trace;
      st->rate_acc = rate_a;
      st->rate_trials = rate_t;
    }
  }

  __syncthreads();
  {
    const int ns = s1 - s0;
#pragma unroll 1
    for (int f = 0; f < M + 1; ++f) {              // (the labels do not change)
      if (f < M && f >= a.C) continue;
#pragma unroll 1
      for (int nl = tid; nl < ns; nl += kLoopThreads)
        a.srec[(size_t)(f < M ? f : kRecLoss) * a.Np + s0 + nl] = R.at(nl, f);
    }
  }
}

// ------------------------------------------------------------------------------------------------
// Explicit candidates (mca_eval_candidates, mca_eval_trials): loss changes against the current state,
// no commit. CTA r evaluates every candidate on its range, warp per sub-chunk, and the last CTA to
// finish adds the ranges' partials in range order and writes the results. What bounds it is latency:
// one chain of dependent loads (candidate, CSR entries, hidden fields), so 32 warps a CTA keep up to 32
// sub-chunks in flight, and no CTA waits for another (the trial loop's explicit mode, a cooperative
// launch of 16 warps with a grid barrier, serves ranges whose records do not fit in shared memory).
// With that mode and two copies back, 16 trials of 784-64-10 on 1000 samples took 65 us and 64 candidates
// of 784-16384-10 on 60000 samples 58 us of host time; now 23 and 33 us.
// ------------------------------------------------------------------------------------------------
constexpr int kEvalThreads = 1024;
constexpr int kEvalWarps = kEvalThreads / 32;

template <int ACT1, int ACT2, int LOSS, int M>
__global__ void __launch_bounds__(kEvalThreads, 1) mlp2_eval_kernel(Mlp2Args a) {
  extern __shared__ __align__(16) float s_dyn[];
  __shared__ Cand s_c[kKmax];
  __shared__ __align__(16) float s_w2c[kKmax][16];
  __shared__ __align__(16) float s_onehot[16][16];
  __shared__ float s_sub[kKmax * kMaxSubs];
  __shared__ int s_total, s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r = blockIdx.x, n = a.n_explicit;
  const int s0 = min(r * a.RS, a.N), s1 = min(s0 + a.RS, a.N), ns = s1 - s0;
  const VRecs<M> R{s_dyn};
  if (tid < n) {
    Cand c;
    fill_candidate(a, a.ex_idx[tid], 0u, true, a.ex_new[tid], r, s0, s1, c);
    c.sub0 = 0;
    s_c[tid] = c;
  }
  // the records (the warps without candidates start with them)
  const int t0 = tid < kKmax ? tid + kEvalThreads - kKmax : tid - kKmax;
#pragma unroll 4
  for (int e = t0; e < (M + 2) * 32 * ((ns + 31) / 32); e += kEvalThreads) {
    const int f = (e >> 5) % (M + 2), nl = (e >> 5) / (M + 2) * 32 + lane;
    if (nl < ns)
      R.at(nl, f) = f < M && f >= a.C
                        ? -INFINITY
                        : a.srec[(size_t)(f < M ? f : f - M + kRecLoss) * a.Np + s0 + nl];
  }
  if (tid < 256) s_onehot[tid >> 4][tid & 15] = (tid >> 4) == (tid & 15) ? -1.0f : 0.0f;
  __syncthreads();
  for (int e = tid; e < n * 16; e += kEvalThreads) {
    const Cand& c = s_c[e >> 4];
    const int q = e & 15;
    s_w2c[e >> 4][q] =
        c.layer == 0 && c.gcnt > 0 && q < a.C ? a.w2[(size_t)q * a.H + c.row] : 0.0f;
  }
  if (warp == 0) {                   // exclusive scan of the sub-chunk counts, four candidates a lane
    int v[4], loc = 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      v[t] = lane * 4 + t < n ? s_c[lane * 4 + t].nsub : 0;
      loc += v[t];
    }
    int inc = loc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    int ex = inc - loc;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (lane * 4 + t < n) s_c[lane * 4 + t].sub0 = ex;
      ex += v[t];
    }
    if (lane == 31) s_total = inc;
  }
  __syncthreads();
  {
    int k = 0;
#pragma unroll 1
    for (int it = warp; it < s_total; it += kEvalWarps) {
      while (s_c[k].sub0 + s_c[k].nsub <= it) ++k;
      const Cand& c = s_c[k];
      const int e_lo = (it - c.sub0) * a.SUB, e_hi = min(e_lo + a.SUB, c.ecnt);
      const float* zrow = a.z1 + (size_t)(c.layer == 0 ? c.row : c.col) * a.Np;
      const Direction<M> dir = direction<M>(c, s_w2c[k]);
      float acc = 0.0f;
#pragma unroll 1
      for (int g = e_lo; g < e_hi; g += 96) {      // three entries' loads in flight per lane
        int nn[3];
        float xv[3], zv[3];
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          const int e = g + t * 32 + lane;
          nn[t] = -1;
          xv[t] = 0.0f;
          if (e < e_hi) {
            nn[t] = c.layer == 0 ? __ldg(a.xs_n + c.ebeg + e) : s0 + e;
            if (c.layer == 0) xv[t] = __ldg(a.xs_v + c.ebeg + e);
          }
        }
#pragma unroll
        for (int t = 0; t < 3; ++t) zv[t] = nn[t] >= 0 ? zrow[nn[t]] : 0.0f;
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          float zn;
          const float da = entry_step<ACT1>(a, c, xv[t], zv[t], zn);
          if (nn[t] >= 0)
            acc += vdelta<ACT2, LOSS, M, false>(a, R, &s_onehot[0][0], dir, nn[t] - s0,
                                                       da);
        }
      }
      __syncwarp();
      acc = warp_sum(acc);
      if (lane == 0) s_sub[it] = acc;
    }
  }
  __syncthreads();
  for (int k = tid; k < n; k += kEvalThreads) {
    float s = 0.0f;
    const int b = s_c[k].sub0, nb = s_c[k].nsub;
    for (int q = 0; q < nb; ++q) s += s_sub[b + q];
    a.partial[(size_t)k * a.NR + r] = s;
  }
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    s_last = atomicAdd(&a.bar->count, 1u) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  if (!s_last) return;
  for (int k = warp; k < n; k += kEvalWarps) {
    float hi = 0.0f, lo = 0.0f;
    for (int q = lane; q < a.NR; q += 32)
      two_sum_add(hi, lo, s_c[k].gcnt > 0 ? __ldcg(a.partial + (size_t)k * a.NR + q) : 0.0f);
    const float t = warp_sum_comp(hi, lo);
    if (lane == 0) a.ex_out[k] = s_c[k].valid ? (double)t : __longlong_as_double(0x7ff8000000000000ll);
  }
  if (tid == 0) {
    a.bar->count = 0u;               // ready for the next launch
    if (a.ex_tail != nullptr) {
      a.ex_tail->S = a.st->S;
      a.ex_tail->err = a.st->err;
    }
  }
}

// Trial-loop and evaluation kernels by hidden transfer function and class count C, for sigmoid outputs
// with MSE (mca_mlp2_mse.cu) and identity outputs with cross-entropy (mca_mlp2_ce.cu).
using LoopFn = void (*)(Mlp2Args);
enum LoopKind { kLoopTrial, kLoopWindow, kLoopEval };
LoopFn loop_variant_mse(LoopKind kind, int act1, int C);
LoopFn loop_variant_ce(LoopKind kind, int act1, int C);

template <int ACT1, int ACT2, int LOSS, int NC, int M>
LoopFn loop_kernel(LoopKind kind) {
  return kind == kLoopEval     ? mlp2_eval_kernel<ACT1, ACT2, LOSS, M>
         : kind == kLoopWindow ? mlp2_window_loop<ACT1, ACT2, LOSS, M>
                               : mlp2_trial_loop<ACT1, ACT2, LOSS, NC>;
}

template <int ACT2, int LOSS, int NC, int M>
LoopFn loop_variant(LoopKind kind, int act1) {
  switch (act1) {
    case MCA_ACT_TANH: return loop_kernel<MCA_ACT_TANH, ACT2, LOSS, NC, M>(kind);
    case MCA_ACT_GAUSSIAN: return loop_kernel<MCA_ACT_GAUSSIAN, ACT2, LOSS, NC, M>(kind);
    case MCA_ACT_RELU: return loop_kernel<MCA_ACT_RELU, ACT2, LOSS, NC, M>(kind);
    default: return loop_kernel<-1, ACT2, LOSS, NC, M>(kind);
  }
}

}  // namespace mca

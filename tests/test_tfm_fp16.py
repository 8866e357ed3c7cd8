"""The Transformer kernels with fp16 operand parts: the range rule that chooses them (needs a GPU), and
their weight images in the order of consumption (CPU).

Tolerances: dS within TIE_REL * S of the fp64 oracle, as everywhere (parity.py)."""
import dataclasses
import os
import subprocess

import numpy as np
import pytest

from oracle import mca_tfm as T
from paper_2607_08406_gb300 import workloads as W

from parity import TIE_REL, compare, forced_from_oracle

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.gpu
@pytest.mark.parametrize("layers,ff,vocab", [(1, 128, 2), (2, 384, 128), (3, 1024, 65)])
@pytest.mark.parametrize("big", [1.0, 4.0, 30.0])
def test_tfm_parameter_range(gpu_lib, layers, ff, vocab, big):
    """Parameters up to `big`: the fp16 kernels up to 4, the tf32 kernels beyond; explicit candidates
    of either size in every parameter tensor; the smallest and largest feed-forward width and
    vocabulary. Both sides of the range answer alike."""
    spec = W.TfmSpec(vocab=vocab, n_layer=layers, d_ff=ff)
    wl = W.char_transformer(batch=2, text_len=4000, spec=spec, n_trials=8, K=8)
    rng = np.random.default_rng(5)
    init = wl.init.copy()
    init[rng.integers(0, init.size, 40)] = rng.uniform(-1, 1, 40).astype(np.float32)
    init[rng.integers(0, init.size)] = np.float32(big)
    wl.init = init
    h = gpu_lib.create_from_tfm_workload(wl)
    assert gpu_lib.mca_get_stats(h)["tensor_cores"] == 1
    flat = init.astype(np.float64)
    S0 = T.tfm_seq_losses(spec, flat, wl.tokens).sum()
    assert gpu_lib.mca_loss(h) * 2 * spec.ctx == pytest.approx(S0, rel=TIE_REL)
    idx, o = [], 0
    for _, shape in spec.blocks():
        n = int(np.prod(shape))
        idx.append(o + int(rng.integers(0, n)))
        o += n
    idx = np.array(idx[:128], np.uint32)
    for amp in (1.0, 8.0):
        new = rng.uniform(-amp, amp, len(idx)).astype(np.float32)
        got = gpu_lib.mca_eval_candidates(h, idx, new)
        for i, v, d in zip(idx, new, got):
            old, flat[i] = flat[i], v
            want = T.tfm_seq_losses(spec, flat, wl.tokens).sum() - S0
            flat[i] = old
            assert abs(d - want) <= TIE_REL * max(S0, S0 + want)


def _growing(n, top=3.5, delta=0.45):
    """A perturbing workload whose largest parameters grow past 4 - delta within n trials: some at
    +-top."""
    spec = W.TfmSpec(n_layer=1, d_ff=128)
    wl = W.char_transformer(batch=2, text_len=4000, spec=spec, n_trials=n, K=8)
    wl.domain = dataclasses.replace(wl.domain, op="perturb", delta=delta)
    rng = np.random.default_rng(2)
    wl.init = wl.init.copy()
    big = rng.random(wl.init.size) < 0.15
    o = 0
    for name, shape in spec.blocks():            # (not the matrices of the attention scores)
        m = int(np.prod(shape))
        if name[-2:] in ("wq", "wk", "bq", "bk"):
            big[o:o + m] = False
        o += m
    wl.init[big] = (top * rng.choice([-1.0, 1.0], big.sum())).astype(np.float32)
    return wl


def _crossing(tr, init, domain):
    """Trials ahead of which the largest parameter plus a step lies within 4, and accepted trials
    on either side."""
    top = float(np.abs(init).max())
    inside = []
    for k in range(len(tr["tau"])):
        inside.append(top + domain.delta <= 4.0)
        if tr["accept"][k]:
            top = max(top, abs(float(np.float32(tr["new"][k]))))
    inside = np.array(inside)
    return inside, tr["accept"] & inside, tr["accept"] & ~inside


@pytest.mark.gpu
@pytest.mark.parametrize("period", [0, 25])
def test_tfm_perturbations_leave_the_fp16_range(gpu_lib, period):
    """A run whose parameters grow past the fp16 kernels' bound continues on the tf32 kernels: with
    batches enqueued one ahead, and in round trips (resync period). Accepted trials on both sides."""
    n = 60
    wl = _growing(n)
    tr, flat, S = T.run_full_tfm(wl.spec, wl.tokens, wl.init, n, 1, wl.domain)
    inside, before, after = _crossing(tr, wl.init, wl.domain)
    assert 3 <= inside.sum() <= n - 20 and before.sum() >= 2 and after.sum() >= 5
    h = gpu_lib.create_from_tfm_workload(wl, trace_cap=n, resync_period=period)
    gpu_lib.mca_force_decisions(h, *forced_from_oracle(tr))
    st = gpu_lib.mca_run(h, n, 1)
    assert st["resyncs"] == 1 + (n // period if period else 0)        # one for the change of kernels
    compare(gpu_lib.mca_get_trace(h, n), tr)
    assert np.array_equal(gpu_lib.mca_get_params(h, wl.n_params), flat)
    cached = gpu_lib.mca_loss(h)
    gpu_lib.mca_resync(h)
    assert gpu_lib.mca_loss(h) == pytest.approx(cached, rel=TIE_REL)


@pytest.mark.gpu
@pytest.mark.parametrize("top,delta", [(3.5, 0.45), (3.05, 0.45), (0.9, 0.15), (0.05, 0.8)])
def test_tfm_trajectory_does_not_depend_on_the_batch_width(gpu_lib, top, delta):
    """Perturbed parameters that cross 4 (fp16 to tf32 kernels) or powers of two below (the operands' scales)
    on the way: the same trace, bit for bit, for every batch width and split of the run."""
    n = 120
    wl = _growing(n, top, delta)
    out = []
    for K, fixed, parts in ((1, True, (n,)), (16, True, (n,)), (5, False, (n,)), (64, False, (7, 40, n - 47))):
        h = gpu_lib.create_from_tfm_workload(wl, trace_cap=n, K=K, fixed_K=fixed)
        for m in parts:
            gpu_lib.mca_run(h, m, 3)
        out.append((gpu_lib.mca_get_trace(h, n), gpu_lib.mca_get_params(h, wl.n_params),
                    gpu_lib.mca_loss(h)))
    assert out[0][0]["accept"].sum() > 10
    for o in out[1:]:
        assert np.array_equal(o[0], out[0][0])
        assert np.array_equal(o[1], out[0][1]) and o[2] == out[0][2]


@pytest.mark.gpu
def test_tfm_growing_feed_forward_activation(gpu_lib):
    """exp(-g u^2) with g < 0 has no bound that the fp16 operands could hold."""
    spec = W.TfmSpec(n_layer=1, d_ff=128, act="gaussian", act_param=-0.25)
    wl = W.char_transformer(batch=2, text_len=4000, spec=spec, n_trials=8, K=8)
    rng = np.random.default_rng(1)
    wl.init, o = wl.init.copy(), 0
    for name, shape in spec.blocks():
        m = int(np.prod(shape))
        if name == "b0.b1":
            wl.init[o:o + 3] = np.float32(3.0)
        if name == "b0.w1":                          # u up to about 8: activations up to 1e7
            wl.init[o:o + m] = rng.normal(0.0, 0.2, m)
        if name == "b0.w2":
            wl.init[o:o + m] = rng.normal(0.0, 1e-3, m)
        o += m
    flat = wl.init.astype(np.float64)
    S0 = T.tfm_seq_losses(spec, flat, wl.tokens).sum()
    h = gpu_lib.create_from_tfm_workload(wl)
    assert gpu_lib.mca_get_stats(h)["tensor_cores"] == 1
    assert gpu_lib.mca_loss(h) * 2 * spec.ctx == pytest.approx(S0, rel=TIE_REL)


@pytest.mark.gpu
@pytest.mark.parametrize("v", [1e-2, 1e-3, 1e-4, 1e-5, 1e-6])
def test_tfm_small_activations(gpu_lib, v):
    """Attention outputs and feed-forward activations of size v that the residual stream consists of (tiny
    embeddings, an epsilon below the stream's variance): in fp16 parts or, if those lose bits, in tf32 parts."""
    spec = W.TfmSpec(n_layer=1, d_ff=128, ln_eps=1e-30)
    wl = W.char_transformer(batch=2, text_len=4000, spec=spec, n_trials=8, K=8)
    rng = np.random.default_rng(3)
    amp = {"tok_emb": 1e-6 * v, "pos_emb": 1e-6 * v, "b0.wq": 0.05, "b0.wk": 0.05, "b0.wv": v / 4,
           "b0.wo": 0.3, "b0.w1": v / 11, "b0.w2": 0.3, "w_head": 0.5}
    wl.init = np.concatenate([
        (np.ones(shape) if name.endswith(".g") else rng.normal(0.0, amp.get(name, 0.0) or 1e-30, shape)
         ).ravel() for name, shape in spec.blocks()]).astype(np.float32)
    S0 = T.tfm_seq_losses(spec, wl.init.astype(np.float64), wl.tokens).sum()
    h = gpu_lib.create_from_tfm_workload(wl)
    assert gpu_lib.mca_loss(h) * 2 * spec.ctx == pytest.approx(S0, rel=TIE_REL)


PROBE = r"""
#include <cstdio>
#include <cstdlib>
#include "%s"
int main(int, char** argv) {
  const int F = atoi(argv[1]), nL = atoi(argv[2]);
  printf("%%zu\n", mca::tfm_f16_image_bytes(F, nL));
  for (int b = 0; b <= nL; ++b)
    for (int m = 0; m < 7; ++m) {
      if ((b == nL) != (m == mca::kTcHead)) continue;
      const int rows = m == mca::kTcW1 ? F : 128, cols = m == mca::kTcW2 ? F : 128;
      for (int r = 0; r < rows; ++r)
        for (int k = 0; k < cols; ++k)
          printf("%%d %%d %%d %%d %%zu\n", b, m, r, k, mca::tfm_f16_image_offset(m, b, r, k, F, nL));
    }
}
"""


@pytest.mark.parametrize("F,nL", [(128, 1), (512, 2), (1024, 1)])
def test_tfm_f16_image_is_the_order_of_consumption(tmp_path, F, nL):
    """Chunk by chunk as the control warp issues the MMAs, each chunk the canonical K-major layout (8
    rows x 16 bytes core matrices, K groups of 8 columns after another), hi then lo."""
    header = os.path.join(ROOT, "paper_2607_08406_gb300", "csrc", "mca_tc_layout.h")
    (tmp_path / "p.cpp").write_text(PROBE % header)
    subprocess.run(["g++", "-std=c++17", "-O1", str(tmp_path / "p.cpp"), "-o", str(tmp_path / "p")],
                   check=True)
    out = subprocess.run([str(tmp_path / "p"), str(F), str(nL)], capture_output=True, text=True,
                         check=True).stdout.split("\n")
    got = np.array([list(map(int, x.split())) for x in out[1:] if x])
    want, chunk = {}, 0

    def put(b, m, r0, rows, k0, cols):
        nonlocal chunk
        for r in range(rows):
            for k in range(cols):
                o = chunk * 8192 + (k // 8) * rows * 8 + r * 8 + k % 8
                want[(b, m, r0 + r, k0 + k)] = o
        chunk += 1

    n = F // 64
    for b in range(nL):
        for m in range(4):
            for q in range(4):
                put(b, m, 0, 128, 32 * q, 32)

        def w1(h):
            for q in range(2):
                put(b, 4, 64 * h, 64, 64 * q, 64)

        w1(0), w1(1)
        for h in range(n):
            for q in range(2):
                put(b, 5, 0, 128, 64 * h + 32 * q, 32)
            if h + 2 < n:
                w1(h + 2)
    for q in range(4):
        put(nL, 6, 0, 128, 32 * q, 32)
    assert int(out[0]) == chunk * 16384
    assert len(got) == len(want)
    assert all(want[tuple(g[:4])] == g[4] for g in got.tolist())
    # every high part's low part (4096 elements on) is in the same chunk and is no high part
    offs = np.sort(got[:, 4])
    assert np.all(offs % 8192 < 4096) and len(np.unique(offs)) == len(offs)

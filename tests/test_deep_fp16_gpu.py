"""The deep chain with fp16 operand parts (needs a GPU): weights of any size, and weights that outgrow the
scale of their operands. Tolerance: dS within TIE_REL * S of the fp64 oracle (parity.py)."""
import dataclasses

import numpy as np
import pytest

from oracle import mca_oracle as O
from paper_2607_08406_gb300 import workloads as W

from parity import TIE_REL, compare, forced_from_oracle, oracle_trace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale,delta", [(1.0, 0.75), (1e-3, 2e-3), (40.0, 30.0)])
def test_deep_perturbations_beyond_the_operand_scale(gpu_lib, scale, delta):
    """Perturbed weights outgrow the bound their fp16 images were scaled for: the images are split
    again. Tiny and large weights, three layers (one dense) and a ragged tile."""
    wl = W.mlp_deep(N=300, width=256, depth=3, n_trials=120, K=16)
    wl.init = (wl.init * np.float32(scale)).astype(np.float32)
    wl.domain = dataclasses.replace(wl.domain, op="perturb", delta=delta)
    tr, params, S = oracle_trace(wl, 120)
    h = gpu_lib.create_from_workload(wl, trace_cap=120)
    gpu_lib.mca_force_decisions(h, *forced_from_oracle(tr))
    st = gpu_lib.mca_run(h, 120, wl.seed)
    assert st["tensor_cores"] == 1 and st["accepts"] > 10
    compare(gpu_lib.mca_get_trace(h, 120), tr)
    assert np.array_equal(gpu_lib.mca_get_params(h, wl.n_params), params.flat_eff32())
    cached = gpu_lib.mca_loss(h)
    gpu_lib.mca_resync(h)
    assert gpu_lib.mca_loss(h) == pytest.approx(cached, rel=TIE_REL)
    assert cached == pytest.approx(S / wl.N, rel=TIE_REL)


def _check_candidates(gpu_lib, wl, h, new_amp=1.0, n=32):
    """dS of n candidates in the layers ahead of a dense one, against the fp64 oracle."""
    flat = gpu_lib.mca_get_params(h, wl.n_params)
    rng = np.random.default_rng(11)
    off = np.cumsum([0] + [ly.n_in * ly.n_out for ly in wl.layers])
    idx = np.concatenate([rng.integers(off[0], off[1], n // 2),
                          rng.integers(off[1], off[2], n // 2)]).astype(np.uint32)
    new = rng.uniform(-new_amp, new_amp, n).astype(np.float32)
    got = gpu_lib.mca_eval_candidates(h, idx, new)
    X = wl.X.T.astype(np.float64)

    def total(f):
        return O.total_loss(O.Params(wl.layers, f), X, wl.y, wl.loss)

    S = total(flat)
    for k in range(n):
        f = flat.copy()
        f[idx[k]] = new[k]
        want = total(f) - S
        assert abs(got[k] - want) <= TIE_REL * max(S, S + want), k
    return got


def test_channel_call_without_trials_changes_nothing(gpu_lib):
    """The operands' scale may only grow together with the images: a channel call with no trials on
    weights below the He amplitude leaves every loss change as it was."""
    wl = W.mlp_deep(N=300, width=256, depth=4, n_trials=16, K=16)
    wl.domain = dataclasses.replace(wl.domain, op="perturb", delta=0.01)
    h = gpu_lib.create_from_workload(wl)
    before = _check_candidates(gpu_lib, wl, h)
    for scheme in ("he", "zero"):
        acc, dS = gpu_lib.mca_run_channels(h, 0, 3, scheme)
        assert len(acc) == 0 and len(dS) == 0
        assert np.array_equal(_check_candidates(gpu_lib, wl, h), before)
    gpu_lib.mca_run_channels(h, 3, 3, "he")
    _check_candidates(gpu_lib, wl, h)


@pytest.mark.parametrize("case", ["outlier", "domain", "perturb_outlier", "he_over_tiny"])
def test_deep_weights_of_a_wide_range(gpu_lib, case):
    """Weights far below the scale of the fp16 operands (one huge dense weight, a wide replacement domain,
    a step that makes one weight huge, He values over tiny weights) take the tf32 parts."""
    wl = W.mlp_deep(N=300, width=256, depth=4, n_trials=16, K=16)
    dense = wl.layers[0].n_in * 256
    if case == "outlier":
        wl.init[dense + 256 * 7 + 3] = np.float32(1e10)
        wl.domain = dataclasses.replace(wl.domain, op="perturb", delta=0.01)
        h = gpu_lib.create_from_workload(wl)
    elif case == "domain":
        wl.domain = dataclasses.replace(wl.domain, lo=-2.0 ** 31, hi=2.0 ** 31)
        h = gpu_lib.create_from_workload(wl)
    elif case == "perturb_outlier":
        wl.domain = dataclasses.replace(wl.domain, op="perturb", delta=1e11)
        h = gpu_lib.create_from_workload(wl, trace_cap=40)
        tau = np.arange(40, dtype=np.uint64)
        gpu_lib.mca_force_decisions(h, tau, tau % 2 == 0)
        gpu_lib.mca_run(h, 40, 3)
        moved = np.abs(gpu_lib.mca_get_params(h, wl.n_params)[dense:dense + 256 * 256 * 3]) > 1e8
        assert moved.any()
    else:
        wl.init = (wl.init * np.float32(2.0 ** -30)).astype(np.float32)
        wl.init[:dense] *= np.float32(2.0 ** 30)
        wl.domain = dataclasses.replace(wl.domain, op="perturb", delta=2.0 ** -31)
        h = gpu_lib.create_from_workload(wl)
        gpu_lib.mca_force_decisions(h, [0, 1], [True, False])
        gpu_lib.mca_run_channels(h, 2, 5, "he")
        st = gpu_lib.mca_get_params(h, wl.n_params)
        assert (np.abs(st[dense:dense + 256 * 256 * 3]) > 1e-4).sum() == 3
    assert gpu_lib.mca_get_stats(h)["tensor_cores"] == 1
    _check_candidates(gpu_lib, wl, h)
    cached = gpu_lib.mca_loss(h)
    gpu_lib.mca_resync(h)
    assert gpu_lib.mca_loss(h) == pytest.approx(cached, rel=TIE_REL)


@pytest.mark.parametrize("kind", ["deep", "tfm"])
def test_resume_where_a_large_weight_has_gone(gpu_lib, kind):
    """A run that starts with one large weight (tf32 parts of the deep chain, a larger scale of the
    Transformer's operands), which an accepted trial replaces: from the next resync on it is the run
    that mca_set_params starts from the parameters there, bit for bit."""
    n, period = 60, 20
    if kind == "deep":
        wl = W.mlp_deep(N=300, width=256, depth=4, n_trials=n, K=8)
        lo, hi, big = 784 * 256, 784 * 256 + 3 * 65536, 1e10
        create = gpu_lib.create_from_workload
    else:
        wl = W.char_transformer(batch=2, text_len=4000, n_trials=n, K=8,
                                spec=W.TfmSpec(n_layer=1, d_ff=128))
        lo, hi, big = 0, wl.n_params, 4.0
        create = gpu_lib.create_from_tfm_workload
    seed = 2
    h = create(wl, trace_cap=n)
    gpu_lib.mca_run(h, n, seed)
    tr = gpu_lib.mca_get_trace(h, n)[:period]
    k = int(np.flatnonzero((tr["idx"] >= lo) & (tr["idx"] < hi))[0])
    wl.init = wl.init.copy()
    wl.init[tr["idx"][k]] = np.float32(big)
    full = create(wl, trace_cap=n, resync_period=period)
    gpu_lib.mca_force_decisions(full, [k], [True])
    gpu_lib.mca_run(full, n, seed)
    part = create(wl, trace_cap=n, resync_period=period)
    gpu_lib.mca_force_decisions(part, [k], [True])
    gpu_lib.mca_run(part, period, seed)
    params = gpu_lib.mca_get_params(part, wl.n_params)
    assert np.abs(params[lo:hi]).max() < 2.0
    again = create(wl, trace_cap=n, resync_period=period)
    gpu_lib.mca_set_params(again, params, tau=period)
    gpu_lib.mca_run(again, n - period, seed)
    assert np.array_equal(gpu_lib.mca_get_trace(again, n), gpu_lib.mca_get_trace(full, n)[period:])
    assert gpu_lib.mca_loss(again) == gpu_lib.mca_loss(full)
    gpu_lib.mca_resync(part)
    gpu_lib.mca_run(part, n - period, seed)
    assert gpu_lib.mca_loss(part) == gpu_lib.mca_loss(full)

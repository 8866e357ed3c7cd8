"""Explicit evaluation (mca_eval_candidates, mca_eval_trials) of single-hidden-layer nets (needs a GPU):
both record sizes, one to 128 candidates, features without entries, unchanged weights, and the
explicit mode of the trial loop for ranges whose records do not fit in shared memory (grid = 1).

Tolerances: dS within TIE_REL * S of the fp64 oracle, as everywhere (parity.py)."""
import numpy as np
import pytest

from oracle import mca_oracle as O
from paper_2607_08406_gb300 import workloads as W

from parity import TIE_REL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,hidden,out,loss,N,H,n,grid", [
    (2, "relu", "identity", "softmax_ce", 9, 2, 1, 0),
    (7, "gaussian", "sigmoid", "mse_onehot", 1003, 5, 31, 0),
    (10, "tanh", "identity", "softmax_ce", 30011, 64, 128, 0),
    (11, "tanh", "sigmoid", "mse_onehot", 2999, 8, 64, 0),
    (14, "gelu", "identity", "softmax_ce", 20003, 16, 127, 0),
    (10, "tanh", "identity", "softmax_ce", 5003, 16, 33, 1),
])
def test_explicit_candidates(gpu_lib, C, hidden, out, loss, N, H, n, grid):
    D = 40
    rng = np.random.default_rng(N)
    layers = [W.Layer(D, H, hidden, 0.7), W.Layer(H, C, out)]
    X = W.synth_images(rng, N, D, 0.4)
    X[:, 3] = 0.0                                     # a feature without entries
    wl = W.MLPWorkload("explicit", layers, loss, X, rng.integers(0, C, N).astype(np.int32),
                       W.uniform_init(rng, layers, 0.3), 50, 16)
    h = gpu_lib.create_from_workload(wl, grid=grid)
    X64, P1 = wl.X.T.astype(np.float64), D * H

    def total(flat):
        return O.total_loss(O.Params(layers, flat), X64, wl.y, loss)

    for rep in range(2):                              # again after a run has moved the state
        flat = gpu_lib.mca_get_params(h, wl.n_params)
        idx = np.concatenate([rng.integers(P1, wl.n_params, n // 2),
                              rng.integers(0, P1, n - n // 2)]).astype(np.uint32)
        new = rng.uniform(-1, 1, n).astype(np.float32)
        idx[-1] = 3                                   # reads the feature without entries
        if n > 2:
            new[0], new[-2] = flat[idx[0]], flat[idx[-2]]
        got = gpu_lib.mca_eval_candidates(h, idx, new)
        S = total(flat)
        assert got[-1] == 0.0
        if n > 2:
            assert got[0] == 0.0 and got[-2] == 0.0
        check = range(n) if N < 5000 else range(0, n, 9)
        for k in check:
            f = flat.copy()
            f[idx[k]] = new[k]
            want = total(f) - S
            assert abs(got[k] - want) <= TIE_REL * max(S, S + want), k
        rec = gpu_lib.mca_eval_trials(h, wl.seed + 5, 77, min(n, 16))
        again = gpu_lib.mca_eval_candidates(h, rec["idx"].astype(np.uint32), rec["new_w"])
        assert np.array_equal(rec["dS"].astype(np.float64), again)
        assert np.all(np.abs(rec["S"] - S) <= TIE_REL * S)
        gpu_lib.mca_run(h, 50, wl.seed)


@pytest.mark.parametrize("C,hidden,out,loss", [
    (10, "tanh", "identity", "softmax_ce"),
    (10, "tanh", "sigmoid", "mse_onehot"),
    (7, "gaussian", "sigmoid", "mse_onehot"),
    (13, "relu", "identity", "softmax_ce"),
    (10, "gelu", "tanh", "mse_onehot"),
])
def test_changes_that_reach_no_output_field_are_zero(gpu_lib, C, hidden, out, loss):
    """A hidden neuron without outgoing weights: its activation changes, no output field does, and the loss
    change is exactly 0 (a neutral trial), in the evaluation kernel and in the windowed loop, before
    and after commits."""
    N, D, H = 3001, 20, 9
    rng = np.random.default_rng(C)
    layers = [W.Layer(D, H, hidden, 0.7), W.Layer(H, C, out)]
    init = W.uniform_init(rng, layers, 0.3)
    init[D * H:].reshape(C, H)[:, ::2] = 0.0            # neurons 0, 2, ..: no outgoing weight
    wl = W.MLPWorkload("neutral", layers, loss, W.synth_images(rng, N, D, 0.4),
                       rng.integers(0, C, N).astype(np.int32), init, 300, 16)
    h = gpu_lib.create_from_workload(wl, trace_cap=300)
    idx = np.array([j * D + i for j in range(0, H, 2) for i in range(0, D, 3)], np.uint32)
    new = rng.uniform(-1, 1, len(idx)).astype(np.float32)
    assert np.all(gpu_lib.mca_eval_candidates(h, idx, new) == 0.0)
    gpu_lib.mca_run(h, 300, 5)
    tr = gpu_lib.mca_get_trace(h, 300)
    live = init[D * H:].reshape(C, H) != 0.0
    seen = 0
    for t in tr:
        i = int(t["idx"])
        if i < D * H:
            if not live[:, i // D].any():
                assert t["dS"] == 0.0 and t["accept"] == 1
                seen += 1
        elif t["accept"]:
            live[(i - D * H) // H, (i - D * H) % H] = t["new_w"] != 0.0
    assert seen > 15 and tr["accept"].sum() > 60
    got = gpu_lib.mca_get_params(h, wl.n_params)[D * H:].reshape(C, H)
    dead = [j for j in range(H) if not got[:, j].any()]
    idx = np.array([j * D + 1 for j in dead], np.uint32)
    if dead:
        assert np.all(gpu_lib.mca_eval_candidates(h, idx, np.full(len(idx), 0.9, np.float32)) == 0.0)

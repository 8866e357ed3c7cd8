"""Sample records of the windowed trial loop (needs a GPU): both record sizes (up to 10 and up to 14
classes) with and without unused fields, every compiled combination of transfer function and loss, and
hidden fields that overflow.

Tolerances: dS within TIE_REL * S of the fp64 oracle, as everywhere (parity.py)."""
import numpy as np
import pytest

from oracle import mca_oracle as O
from paper_2607_08406_gb300 import workloads as W

from parity import TIE_REL, compare, forced_from_oracle, oracle_trace

pytestmark = pytest.mark.gpu


def _net(C, hidden, out, loss, N, H, D=60, beta=float("inf"), hi=1.0):
    rng = np.random.default_rng(C * 1000 + N)
    layers = [W.Layer(D, H, hidden, 0.7), W.Layer(H, C, out)]
    return W.MLPWorkload("records", layers, loss, W.synth_images(rng, N, D, 0.4),
                         rng.integers(0, C, N).astype(np.int32), W.uniform_init(rng, layers, 0.3),
                         600, 16, domain=W.Domain(lo=-hi, hi=hi, beta=beta))


@pytest.mark.parametrize("C,hidden,out,loss,N,H,beta", [
    (2, "tanh", "sigmoid", "mse_onehot", 517, 3, float("inf")),
    (3, "relu", "identity", "softmax_ce", 1201, 16, float("inf")),
    (9, "gaussian", "identity", "softmax_ce", 1003, 8, float("inf")),
    (10, "gelu", "sigmoid", "mse_onehot", 1000, 8, float("inf")),
    (10, "tanh", "identity", "softmax_ce", 5003, 16, 3000.0),
    (11, "gaussian", "sigmoid", "mse_onehot", 1999, 8, float("inf")),
    (14, "tanh", "identity", "softmax_ce", 2500, 5, float("inf")),
    (14, "sigmoid", "sigmoid", "mse_onehot", 777, 8, float("inf")),
    (4, "tanh", "tanh", "mse_onehot", 900, 8, float("inf")),
])
def test_record_classes(gpu_lib, C, hidden, out, loss, N, H, beta):
    wl = _net(C, hidden, out, loss, N, H, beta=beta)
    tr, params, S = oracle_trace(wl, wl.n_trials)
    assert tr["accept"].sum() > 20
    theta = 0.0 if np.isinf(beta) else O.metropolis_threshold(wl.seed, tr["tau"], beta, wl.N)
    # exact zeros are replayed too: a ReLU within rounding of its kink can move in fp32 alone
    band = tr["valid"] & (np.abs(tr["dS"] - theta) < TIE_REL * np.abs(tr["S"]))
    h = gpu_lib.create_from_workload(wl, trace_cap=wl.n_trials)
    gpu_lib.mca_force_decisions(h, tr["tau"][band].astype(np.uint64), tr["accept"][band])
    gpu_lib.mca_run(h, wl.n_trials, wl.seed)
    compare(gpu_lib.mca_get_trace(h, wl.n_trials), tr)
    assert np.array_equal(gpu_lib.mca_get_params(h, wl.n_params), params.flat_eff32())
    assert gpu_lib.mca_loss(h) == pytest.approx(S / wl.N, rel=TIE_REL)


@pytest.mark.parametrize("strict,hi,K", [(False, 1.0, 16), (True, 4.0, 64)])
def test_commit_routes(gpu_lib, strict, hi, K):
    """Ranges of several chunks of entries: candidates whose warps hold every new loss at the commit, and
    (wide batches of many live candidates) those with fewer warps than chunks."""
    wl = _net(10, "tanh", "identity", "softmax_ce", 24000, 6, hi=hi)
    wl.domain.strict, wl.K = strict, K
    n = 400
    tr, params, S = oracle_trace(wl, n)
    assert tr["accept"].sum() >= 20
    h = gpu_lib.create_from_workload(wl, trace_cap=n)
    gpu_lib.mca_force_decisions(h, *forced_from_oracle(tr))
    gpu_lib.mca_run(h, n, wl.seed)
    compare(gpu_lib.mca_get_trace(h, n), tr)
    assert np.array_equal(gpu_lib.mca_get_params(h, wl.n_params), params.flat_eff32())
    cached = gpu_lib.mca_loss(h)
    gpu_lib.mca_resync(h)
    assert gpu_lib.mca_loss(h) == pytest.approx(cached, rel=TIE_REL)


def test_hidden_fields_that_overflow(gpu_lib):
    """An input of 3e38 takes hidden fields to infinity (ReLU), in candidates and then in the state.
    Output weights are positive, so the output fields saturate at +infinity and every loss stays
    finite; fields of 3 unused classes are held beside the 7 used ones."""
    wl = _net(7, "relu", "sigmoid", "mse_onehot", 700, 6, D=8, hi=2.0)
    D, H, C, n = 8, 6, 7, 400
    wl.X[:, 0] = 0.0
    wl.X[::50, 0] = 3e38
    w1, w2 = wl.init[:D * H].reshape(H, D), wl.init[D * H:].reshape(C, H)
    w1[:, 0] = 0.0
    w2[:] = np.abs(w2) + 0.05

    def loss_sum(w1, w2):
        z = np.maximum(wl.X.astype(np.float64) @ w1.T, 0.0) @ w2.T.astype(np.float64)
        p = 0.5 * (1.0 + np.tanh(0.5 * z))
        p[np.arange(wl.N), wl.y] -= 1.0
        return (p * p).sum()

    def run(accept):
        h = gpu_lib.create_from_workload(wl, trace_cap=n)
        tau = np.arange(n, dtype=np.uint64)
        gpu_lib.mca_force_decisions(h, tau, tau == accept)
        gpu_lib.mca_run(h, n, wl.seed)
        return gpu_lib.mca_get_trace(h, n)

    g = run(-1)
    first = (g["idx"] < D * H) & (g["idx"] % D == 0)
    t0 = int(np.nonzero(first & (g["new_w"] > 1.3))[0][0])          # 3e38 * 1.3 overflows
    unit = int(g["idx"][t0]) // D
    for accept in (-1, t0):
        g = run(accept)
        a1, a2 = w1.astype(np.float64), w2.astype(np.float64)
        checked = 0
        for t in range(n):
            i, v = int(g["idx"][t]), float(g["new_w"][t])
            b1, b2 = a1.copy(), a2.copy()
            if i < D * H:
                b1[i // D, i % D] = v
                skip = accept >= 0 and t > accept and i == unit * D     # infinity minus infinity
                skip |= accept >= 0 and t > accept and i // D == unit
            else:
                o, j = (i - D * H) // H, (i - D * H) % H
                b2[o, j] = v
                skip = accept >= 0 and t > accept and j == unit and v < a2[o, j]
            if skip:
                continue
            S = loss_sum(a1, a2)
            want = loss_sum(b1, b2) - S
            assert abs(g["dS"][t] - want) <= TIE_REL * max(S, S + want), (t, i, v)
            checked += 1
            if t == accept:
                a1, a2 = b1, b2
        assert checked > n // 2

"""The SIMT chain of deep nets (needs a GPU): every number of rows per thread (widths up to 64, 128 and
256) at its edges, widths that are no multiple of 4, layers of different widths, tiles of 32 and of 64
samples, and sample counts around a tile.

Tolerances: dS within TIE_REL * S of the fp64 oracle, as everywhere (parity.py)."""
import numpy as np
import pytest

from paper_2607_08406_gb300 import workloads as W

from parity import TIE_REL, compare, oracle_trace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths,N,C,hidden", [
    ((1, 1), 1, 2, "tanh"),
    ((5, 3, 7), 31, 14, "tanh"),
    ((64, 64, 64), 33, 10, "tanh"),
    ((30, 65, 64), 100, 3, "gaussian"),
    ((128, 127, 128), 301, 10, "relu"),
    ((129, 128, 129), 257, 11, "tanh"),
    ((255, 256, 255), 130, 10, "tanh"),
    ((256, 256, 17), 65, 10, "tanh"),
    ((20, 33, 20), 9800, 10, "tanh"),
    ((16, 100, 70), 20001, 5, "tanh"),
    ((16, 200, 70), 10001, 5, "sigmoid"),
])
def test_simt_chain(gpu_lib, widths, N, C, hidden):
    D, n = 24, 90
    rng = np.random.default_rng(N + sum(widths))
    dims = [D, *widths, C]
    layers = [W.Layer(dims[l], dims[l + 1], hidden if l < len(widths) else "identity", 0.4)
              for l in range(len(dims) - 1)]
    init = W.uniform_init(rng, layers, [float(np.sqrt(3.0 / L.n_in)) for L in layers])
    wl = W.MLPWorkload("simt", layers, "softmax_ce", W.synth_images(rng, N, D, 0.5),
                       rng.integers(0, C, N).astype(np.int32), init, n, 16)
    tr, params, S = oracle_trace(wl, n)
    band = tr["valid"] & (np.abs(tr["dS"]) < TIE_REL * np.abs(tr["S"]))
    h = gpu_lib.create_from_workload(wl, trace_cap=n)
    gpu_lib.mca_force_decisions(h, tr["tau"][band].astype(np.uint64), tr["accept"][band])
    st = gpu_lib.mca_run(h, n, wl.seed)
    assert st["tensor_cores"] == 0
    compare(gpu_lib.mca_get_trace(h, n), tr)
    assert np.array_equal(gpu_lib.mca_get_params(h, wl.n_params), params.flat_eff32())
    assert gpu_lib.mca_loss(h) == pytest.approx(S / wl.N, rel=TIE_REL)
    cached = gpu_lib.mca_loss(h)
    gpu_lib.mca_resync(h)
    assert gpu_lib.mca_loss(h) == pytest.approx(cached, rel=TIE_REL)

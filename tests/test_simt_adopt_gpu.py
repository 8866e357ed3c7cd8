"""Adoption of accepted candidates from scratch slots on the SIMT paths (needs a GPU): against the commit
kernels' recomputation (MCA_ADOPT=0), bit for bit, with candidates accepted inside and beyond the 16
slots (fixed batches of 32), in every layer, on ragged tiles of 32 and 64 samples."""
import numpy as np
import pytest

from paper_2607_08406_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _net(widths, N, C):
    rng = np.random.default_rng(N)
    dims = [30, *widths, C]
    layers = [W.Layer(dims[l], dims[l + 1], "tanh" if l < len(widths) else "identity")
              for l in range(len(dims) - 1)]
    init = W.uniform_init(rng, layers, [float(np.sqrt(3.0 / L.n_in)) for L in layers])
    return W.MLPWorkload("adopt", layers, "softmax_ce", W.synth_images(rng, N, 30, 0.5),
                         rng.integers(0, C, N).astype(np.int32), init, 400, 32)


CASES = {
    "narrow": lambda: _net((40, 50, 60, 7), 1003, 5),
    "two_hidden": lambda: _net((9, 11), 333, 14),
    "wide_tiles": lambda: _net((70, 20, 130), 10001, 10),
    "tfm": lambda: W.char_transformer(batch=5, text_len=3000, n_trials=200, K=32,
                                      spec=W.TfmSpec(vocab=31, ctx=19, d_model=48, n_head=3,
                                                     n_layer=2, d_ff=70)),
}


@pytest.mark.parametrize("fixed_K", [False, True])
@pytest.mark.parametrize("case", list(CASES))
def test_simt_adoption_matches_commit(gpu_lib, monkeypatch, case, fixed_K):
    wl = CASES[case]()
    create = gpu_lib.create_from_tfm_workload if case == "tfm" else gpu_lib.create_from_workload
    n = wl.n_trials
    # rejected outright: stretches that carry the acceptances of fixed batches past the slots
    taus = np.arange(n, dtype=np.uint64)
    taus = taus[(taus % 50 >= 10) & (taus % 50 < 35)]
    out = []
    for adopt in (None, "0"):
        if adopt is None:
            monkeypatch.delenv("MCA_ADOPT", raising=False)
        else:
            monkeypatch.setenv("MCA_ADOPT", adopt)
        h = create(wl, trace_cap=n, K=32, fixed_K=fixed_K)
        gpu_lib.mca_force_decisions(h, taus, np.zeros(len(taus), bool))
        st = gpu_lib.mca_run(h, n, 4)
        assert st["tensor_cores"] == 0 and st["accepts"] > 20
        out.append((gpu_lib.mca_get_trace(h, n), gpu_lib.mca_get_params(h, wl.n_params),
                    gpu_lib.mca_loss(h)))
        gpu_lib.mca_resync(h)
        assert gpu_lib.mca_loss(h) == pytest.approx(out[-1][2], rel=1e-5)
        h.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]

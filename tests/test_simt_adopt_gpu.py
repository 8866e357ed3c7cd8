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


@pytest.mark.parametrize("case", ["narrow", "tfm"])
def test_workspace_without_room_for_slots(gpu_lib, monkeypatch, case):
    """The slots of the SIMT paths are taken as far as the caller's workspace reaches: a workspace of the size
    without slots, or with room for some, gives the same run; a smaller one is refused."""
    import torch
    wl = CASES[case]()
    tfm = case == "tfm"
    create = gpu_lib.create_from_tfm_workload if tfm else gpu_lib.create_from_workload

    def size():
        if tfm:
            return gpu_lib.mca_tfm_workspace_size(wl.spec, len(wl.tokens), 32, 200)
        return gpu_lib.mca_workspace_size(wl.layers, wl.loss, wl.X, wl.y, 32, 200)

    full = size()
    monkeypatch.setenv("MCA_ADOPT", "0")
    least = size()
    monkeypatch.delenv("MCA_ADOPT")
    assert least < full
    name = "mca_tfm_workspace_size" if tfm else "mca_workspace_size"
    out = []
    for nbytes in (full, least + (full - least) // 3, least, least - 256):
        with monkeypatch.context() as m:
            m.setattr(gpu_lib, name, lambda *a, **k: nbytes)
            if nbytes < least:
                with pytest.raises(gpu_lib.MCAError, match="workspace"):
                    create(wl, trace_cap=200, K=32)
                continue
            h = create(wl, trace_cap=200, K=32, fixed_K=True)
        gpu_lib.mca_run(h, 200, 4)
        out.append((gpu_lib.mca_get_trace(h, 200), gpu_lib.mca_get_params(h, wl.n_params)))
        h.close()
    assert len(out) == 3
    for o in out[1:]:
        assert np.array_equal(o[0], out[0][0]) and np.array_equal(o[1], out[0][1])

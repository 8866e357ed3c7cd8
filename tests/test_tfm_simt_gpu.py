"""The SIMT Transformer kernel (needs a GPU): head widths on both sides of 32 columns and at the limit of
64, widths that are no multiple of a tile, and the smallest and largest sizes.

Tolerances: dS within TIE_REL * S of the fp64 oracle, as everywhere (parity.py)."""
import numpy as np
import pytest

from oracle import mca_tfm as T
from paper_2607_08406_gb300 import workloads as W

from parity import TIE_REL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab,ctx,d,heads,layers,ff", [
    (2, 1, 1, 1, 1, 1),
    (17, 15, 32, 1, 1, 16),
    (33, 17, 33, 1, 2, 129),
    (50, 48, 96, 2, 1, 200),
    (128, 64, 128, 2, 1, 127),
    (90, 63, 63, 1, 1, 128),
    (65, 33, 124, 31, 1, 130),
])
def test_simt_transformer(gpu_lib, vocab, ctx, d, heads, layers, ff):
    spec = W.TfmSpec(vocab=vocab, ctx=ctx, d_model=d, n_head=heads, n_layer=layers, d_ff=ff)
    wl = W.char_transformer(batch=3, text_len=2000, spec=spec, n_trials=20, K=8)
    rng = np.random.default_rng(d)
    wl.init = (wl.init + rng.uniform(-0.2, 0.2, wl.init.size)).astype(np.float32)
    h = gpu_lib.create_from_tfm_workload(wl)
    assert gpu_lib.mca_get_stats(h)["tensor_cores"] == 0
    flat = wl.init.astype(np.float64)
    S0 = T.tfm_seq_losses(spec, flat, wl.tokens).sum()
    assert gpu_lib.mca_loss(h) * 3 * ctx == pytest.approx(S0, rel=TIE_REL)
    idx, o = [], 0
    for _, shape in spec.blocks():
        n = int(np.prod(shape))
        idx += [o, o + n - 1, o + int(rng.integers(0, n))]
        o += n
    idx = np.array(idx[:128], np.uint32)
    new = rng.uniform(-1, 1, len(idx)).astype(np.float32)
    got = gpu_lib.mca_eval_candidates(h, idx, new)
    for i, v, g in zip(idx, new, got):
        old, flat[i] = flat[i], float(v)
        want = T.tfm_seq_losses(spec, flat, wl.tokens).sum() - S0
        flat[i] = old
        assert abs(g - want) <= TIE_REL * max(S0, S0 + want), i
    gpu_lib.mca_run(h, 20, wl.seed)                   # commits leave what a full recompute gives
    cached = gpu_lib.mca_loss(h)
    gpu_lib.mca_resync(h)
    assert gpu_lib.mca_loss(h) == pytest.approx(cached, rel=TIE_REL)

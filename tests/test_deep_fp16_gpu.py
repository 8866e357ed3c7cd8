"""The deep chain with fp16 operand parts (needs a GPU): weights of any size, and weights that outgrow the
scale of their operands. Tolerance: dS within TIE_REL * S of the fp64 oracle (parity.py)."""
import dataclasses

import numpy as np
import pytest

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

"""The forward SGEMM's tiles (needs a GPU): all three sizes at the edges of their rule, row counts and depths
around a tile and a chunk, with and without a transfer function on the operand.

Tolerance: the loss to 1e-6 of the fp64 oracle (fields summed in fp32 in ascending order)."""
import numpy as np
import pytest

from oracle import mca_oracle as O
from paper_2607_08406_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths,N,D", [
    ((1,), 1, 1),                     # tiles of 32
    ((33,), 1000, 17),
    ((65, 31, 33), 4865, 16),
    ((129,), 6400, 15),               # 150 tiles of 64: still 32
    ((129,), 6600, 33),               # tiles of 64
    ((250, 129), 9000, 40),
    ((257,), 12800, 31),              # 300 tiles of 128: still 64
    ((257,), 13000, 48),              # tiles of 128
    ((129, 200, 130), 19500, 20),
])
def test_forward_loss(gpu_lib, widths, N, D):
    C = 6
    rng = np.random.default_rng(N)
    dims = [D, *widths, C]
    layers = [W.Layer(dims[l], dims[l + 1], "tanh" if l < len(widths) else "identity")
              for l in range(len(dims) - 1)]
    init = W.uniform_init(rng, layers, [float(np.sqrt(3.0 / L.n_in)) for L in layers])
    wl = W.MLPWorkload("sgemm", layers, "softmax_ce", W.synth_images(rng, N, D, 0.5),
                       rng.integers(0, C, N).astype(np.int32), init, 8, 8)
    h = gpu_lib.create_from_workload(wl)
    S = O.total_loss(O.Params(layers, init), wl.X.T.astype(np.float64), wl.y, wl.loss)
    assert gpu_lib.mca_loss(h) == pytest.approx(S / N, rel=1e-6)

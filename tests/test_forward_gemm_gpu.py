"""The forward GEMM's operand forms (needs a GPU): fp16 parts with a scale per row, and tf32 parts for small
products and for rows of a wide range; feature counts around a chunk of 32.

Tolerance: the loss within TIE_REL of the fp64 oracle, as everywhere (parity.py). The tensor cores add
products to their accumulator with truncation, by less than 2^-22 of it per addition of one of the
3 K / 16 (fp16) or 3 K / 8 (tf32) steps, so the fields of 784 features are below 4e-5 of their size off; that
moves the mean loss by 1e-6 here."""
import numpy as np
import pytest

from oracle import mca_oracle as O
from paper_2607_08406_gb300 import workloads as W

from parity import TIE_REL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,D,spread", [
    (22000, 1024, 784, 0.0),          # fp16 parts
    (22000, 1024, 784, 1.0),          # the same, features and weights over 2 decades
    (22000, 1024, 784, 2.0),          # 4 decades: about at the limit of the range rule
    (22000, 1024, 784, 12.0),         # tf32 parts
    (22000, 1024, 799, 0.0),
    (22000, 1024, 801, 0.0),
    (5000, 1024, 33, 0.0),            # below the size rule: tf32 parts
    (130, 256, 5, 12.0),
])
def test_forward_fields(gpu_lib, N, H, D, spread):
    rng = np.random.default_rng(N + D)
    layers = [W.Layer(D, H, "tanh"), W.Layer(H, 10, "identity")]
    c = (10.0 ** rng.uniform(-spread, spread, D)).astype(np.float32)
    X = W.synth_images(rng, N, D, 0.3) * c
    init = W.uniform_init(rng, layers, [float(np.sqrt(3.0 / D)), 0.3])
    init[:H * D] = (init[:H * D].reshape(H, D) / c).ravel()
    X[::97] = 0.0                                     # samples without any feature
    wl = W.MLPWorkload("fields", layers, "softmax_ce", X, rng.integers(0, 10, N).astype(np.int32),
                       init, 8, 8)
    h = gpu_lib.create_from_workload(wl)
    S = O.total_loss(O.Params(layers, init), X.T.astype(np.float64), wl.y, wl.loss)
    assert gpu_lib.mca_loss(h) == pytest.approx(S / N, rel=TIE_REL)


@pytest.mark.parametrize("n_small,down", [(150, 34), (24, 40), (4, 40)])
def test_forward_fields_of_a_few_small_features(gpu_lib, n_small, down):
    """Features far below the others, and hidden units that read only those: a minority of small entries
    in the samples' rows must not lose their bits. Few distinct samples, so that the errors of
    the fields do not average out in the loss."""
    N, H, D = 22000, 256, 784
    rng = np.random.default_rng(n_small)
    layers = [W.Layer(D, H, "tanh"), W.Layer(H, 10, "identity")]
    base = rng.uniform(0.5, 1.0, (4, D)).astype(np.float32)
    base[:, :n_small] *= np.float32(2.0 ** -down)
    X = np.ascontiguousarray(base[np.arange(N) % 4])
    W1 = np.zeros((H, D), np.float32)
    W1[:, :n_small] = rng.uniform(-1, 1, (H, n_small)) * 2.0 ** down / np.sqrt(n_small)
    init = np.concatenate([W1.ravel(), rng.uniform(-0.5, 0.5, H * 10)]).astype(np.float32)
    wl = W.MLPWorkload("fields", layers, "softmax_ce", X, (np.arange(N) % 7).astype(np.int32), init, 8,
                       8)
    h = gpu_lib.create_from_workload(wl)
    S = O.total_loss(O.Params(layers, init), X.T.astype(np.float64), wl.y, wl.loss)
    assert gpu_lib.mca_loss(h) == pytest.approx(S / N, rel=TIE_REL)


def test_forward_last_hidden_field_overflows(gpu_lib):
    """An infinite activation of the last hidden neuron (33 neurons: the rows past it are padding)
    saturates a sigmoid output and nothing else."""
    N, D, H = 70, 5, 33
    rng = np.random.default_rng(0)
    layers = [W.Layer(D, H, "relu"), W.Layer(H, 4, "sigmoid")]
    X = W.synth_images(rng, N, D, 0.6)
    X[:, :2] = 0.0
    X[::9, :2] = 1.0
    init = W.uniform_init(rng, layers, 0.3)
    init[(H - 1) * D:(H - 1) * D + 2] = np.float32(3e38)
    wl = W.MLPWorkload("overflow", layers, "mse_onehot", X, rng.integers(0, 4, N).astype(np.int32),
                       init, 8, 8)
    with np.errstate(over="ignore"):
        S = O.total_loss(O.Params(layers, init), X.T.astype(np.float64), wl.y, wl.loss)
    h = gpu_lib.create_from_workload(wl)
    assert gpu_lib.mca_loss(h) == pytest.approx(S / N, rel=TIE_REL)

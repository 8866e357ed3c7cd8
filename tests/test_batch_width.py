"""The batch width of host-driven batches, compiled for the host, against a search over every width with
the same cost model in fp64 (CPU)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def _value(acc, trials, u, tail, k):
    """Trials consumed by a batch of k candidates, per unit of its cost."""
    p = (acc + 0.5) / (trials + 1.0)
    cost = 0.3 + (max(1.0, k * u) if k * u <= 1.0 else tail + k * u)
    return (1.0 - (1.0 - p) ** k) / cost


def test_width_maximises_trials_per_cost(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "batch_width_host")
    subprocess.run([nvcc, "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2607_08406_gb300", "csrc"), "-o", exe,
                    os.path.join(HERE, "batch_width_host.cu")], check=True, capture_output=True)
    rng = np.random.default_rng(0)
    cases = []
    for _ in range(400):
        trials = float(rng.integers(0, 3000))
        cases.append((float(rng.integers(0, trials + 1)), trials,
                      float(np.float32(2.0 ** rng.uniform(-8, 3))), float(rng.choice([0.7, 0.15])),
                      int(rng.integers(1, 129))))
    cases += [(0.0, 0.0, u, 0.7, 128) for u in (1 / 152, 0.5, 0.999, 1.0, 1.001, 600.0)]
    text = "\n".join(" ".join(repr(v) for v in c) for c in cases)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
    got = [int(v) for v in out.split()]
    assert len(got) == len(cases)
    for c, k in zip(cases, got):
        assert 1 <= k <= c[4]
        best = max(_value(*c[:4], j) for j in range(1, c[4] + 1))
        assert _value(*c[:4], k) >= best * (1 - 1e-5), c     # (equal values: fp32 fractions)
    # a net that leaves most SMs idle takes wider batches, up to the full GPU
    assert got[-6] > got[-5] >= got[-4]

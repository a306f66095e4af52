"""Model A's weight max(phi, 0)^n for every integer exponent that is formed by
products, and for one of each kind that is not, against the FP64 oracle
within the bounds of the short-horizon parity tests (four times the spread of
the FP32 noise model, with floors)."""

import numpy as np
import pytest

from oracle.oracle import OracleSim
from paper_2306_06983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEPS, K, FLOORS = 3, 4.0, (2e-6, 1e-8, 1e-8)


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    from paper_2306_06983_gb300.build import build
    from oracle.oracle import build_oracle
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build()
    build_oracle()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n", [0.5, 1.0, 2.0, 3.0, 4.0, 5.0, 6.0, 7.0, 8.0, 9.0])
@pytest.mark.parametrize("N", [3, 6, 8])
def test_exponent(N, n):
    from paper_2306_06983_gb300.nlbm import Simulation
    p, phi0 = W.random_smooth(64, 48, N, seed=11, model="A", model_a_n=n, n_disks=6)
    phi0 = phi0.astype(np.float32).astype(np.float64)
    a, b = OracleSim(p, phi0), OracleSim(p, phi0, fp32=True)
    a.step(STEPS)
    b.step(STEPS)
    sim = Simulation(p)
    sim.set_phi(phi0)
    sim.step(STEPS)
    got = [t.cpu().numpy().astype(np.float64) for t in sim.moments()]
    sim.close()
    for g, o, o32, floor in zip(got, a.moments(), b.moments(), FLOORS):
        assert np.abs(g - o).max() <= max(floor, K * np.abs(o32 - o).max())

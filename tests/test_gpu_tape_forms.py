"""The taping step as a march and as patches (rows on and off 32-byte sectors,
row windows and per-node pulls): a taped forward ends with the bits of a plain
run, and its sweep gives the same gradients where the segments, and with them
the forms that write the states, are cut differently."""

import numpy as np
import pytest

from paper_2306_06983_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    from paper_2306_06983_gb300.build import build
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("N,model,nx,ny", [(2, "B", 868, 512), (3, "A", 1021, 640), (4, "B", 868, 512), (5, "B", 896, 512),
                                           (5, "B", 1021, 640), (6, "A", 1100, 640), (7, "B", 1021, 640), (8, "A", 744, 512)])
def test_taped_forward_and_sweep(N, model, nx, ny):
    import torch
    from paper_2306_06983_gb300.nlbm import AdjointRun, Simulation
    p, phi0 = W.random_smooth(64, 64, N, seed=N, model=model, n_disks=4)
    p = dict(p, nx=nx, ny=ny, unit_delta=1e-3)
    phi0 = torch.from_numpy(phi0.astype(np.float32)).cuda().repeat(1, ny // 64 + 1, nx // 64 + 1)[:, :ny, :nx].contiguous()
    sim = Simulation(p)
    sim.set_phi(phi0)
    sim.step(4)
    plain = sim.moments()[0]
    sim.close()
    out = []
    for every in (4, 1):   # every step taped by the forward; the last one alone
        run = AdjointRun(p, 4, every)
        phi_T = run.forward(phi0)
        assert torch.equal(phi_T, plain)
        out.append(run.backward(phi_T - 1.0 / N))
        run.close()
    (g0, gs, gm), (h0, hs, hm) = out
    assert torch.equal(g0, h0) and np.array_equal(gs, hs) and gm == hm

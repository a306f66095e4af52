"""dL/dphi_0 of the reverse sweep, node by node, against single reverse steps
chained on the host, on lattices at and off the edges of the sweep's 32 x 8
tiles and beside walls (test_gpu_sweep.py compares the parameter gradients)."""

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


@pytest.mark.parametrize("nx,ny,wall_x,wall_y,N,model", [
    (1, 9, 0, 0, 3, "B"), (31, 7, 0, 0, 2, "A"), (32, 8, 0, 0, 3, "B"), (33, 9, 0, 1, 3, "A"), (34, 17, 1, 0, 4, "B"),
    (4, 4, 1, 1, 3, "B"), (67, 40, 1, 1, 5, "A"), (70, 33, 0, 0, 8, "B"), (96, 9, 1, 1, 6, "B"), (33, 24, 1, 1, 7, "A"),
    (256, 96, 0, 1, 3, "B")])
@pytest.mark.parametrize("n,every", [(1, 1), (5, 2)])
def test_phi0_gradient(nx, ny, wall_x, wall_y, N, model, n, every):
    import torch
    from paper_2306_06983_gb300.nlbm import AdjointRun, Simulation
    p, phi0 = W.random_smooth(nx, ny, N, seed=nx + ny, model=model, wall_x=bool(wall_x), wall_y=bool(wall_y), n_disks=2)
    p["unit_delta"] = 1e-3
    phi0 = phi0.astype(np.float32)
    ns, pl = N - 1, nx * ny
    run = AdjointRun(p, n, every)
    phi_T = run.forward(phi0)
    # a seed with a value of its own at every node
    seed = torch.randn(phi_T.shape, generator=torch.Generator().manual_seed(nx)).cuda()
    g0 = run.backward(seed)[0]
    sim = Simulation(p)
    sim.set_phi(phi0)
    states = []
    for _ in range(n):
        states.append(sim.save().view(torch.float32)[:(10 * ns + 12) * pl].clone())
        sim.step(1)
    sim.close()
    sd = torch.zeros((10 * ns + 12) * pl, dtype=torch.float32, device="cuda")
    sd[(9 * ns + 8) * pl:(10 * ns + 8) * pl] = (seed[:ns] - seed[ns]).reshape(-1)
    for s in reversed(range(n)):
        sd = run.reverse_step(states[s], sd)[0]
    run.close()
    # phi_0 enters step 1 as phi(t - 1) and as the populations f_i = w_i phi_0
    # that it pulls, all of which enter phi with weight 1: the adjoint of the
    # rest population is that of phi at the node
    sd = sd.reshape(10 * ns + 12, ny, nx)
    chained = torch.stack([sd[9 * q] + sd[9 * ns + 8 + q] for q in range(ns)])
    # the two paths' tapes differ in the rounding of their sums: the bound
    # that the parameter gradients are held to
    assert (g0 - chained).abs().max() <= 1e-4 * chained.abs().max()
    assert chained.abs().max() > 0

"""The reverse sweep (population seeds gathered from the step reversed before,
the last segment's tapes kept by the forward) against single reverse steps
chained on the host, on lattices at and off the edges of its 32 x 8 tiles."""

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
    (4, 4, 1, 1, 3, "B"), (67, 40, 1, 1, 5, "A"), (70, 33, 0, 0, 8, "B")])
def test_sweep_matches_single_steps(nx, ny, wall_x, wall_y, N, model):
    import torch
    from paper_2306_06983_gb300.nlbm import AdjointRun, Simulation, pair_list
    p, phi0 = W.random_smooth(nx, ny, N, seed=nx + ny, model=model, wall_x=bool(wall_x), wall_y=bool(wall_y), n_disks=2)
    p["unit_delta"] = 1e-3
    phi0 = phi0.astype(np.float32)
    n, ns, pl = 5, N - 1, nx * ny
    with torch.cuda.stream(torch.cuda.Stream()):
        run = AdjointRun(p, n, 2)
        seed = (run.forward(phi0) - 1.0 / N).contiguous()
        g0, gs, gm = run.backward(seed)
        # again after the same forward (the last segment rebuilt, no graph),
        # and after another forward (the graph replayed)
        for again in (False, True):
            if again:
                run.forward(phi0)
            h0, hs, hm = run.backward(seed)
            assert torch.equal(g0, h0) and np.array_equal(gs, hs) and gm == hm
        sim = Simulation(p)
        sim.set_phi(phi0)
        states = []
        for _ in range(n):
            states.append(sim.save().view(torch.float32)[:(10 * ns + 12) * pl].clone())
            sim.step(1)
        sim.close()
        sd = torch.zeros((10 * ns + 12) * pl, dtype=torch.float32, device=seed.device)
        sd[(9 * ns + 8) * pl:(10 * ns + 8) * pl] = (seed[:ns] - seed[ns]).reshape(-1)
        gs_sum, gm_sum = np.zeros_like(gs), 0.0
        for s in reversed(range(n)):
            sd, g_s, g_m = run.reverse_step(states[s], sd)
            gs_sum += g_s
            gm_sum += g_m
        run.close()
    # the tapes of the two paths differ in the rounding of their sums: the
    # bound of test_taped_sweep_matches_tape_passes
    scale = max(abs(gs[a, b]) for a, b in pair_list(N))
    assert np.abs(gs - gs_sum).max() <= 1e-4 * scale
    assert abs(gm - gm_sum) <= 1e-4 * abs(gm_sum) + 1e-6 * scale

"""The largest lattice that the library accepts (2^28 nodes) with explicit row
marches, with and without row windows.  The library's own choice there, which
test_gpu_max_lattice.py runs against the oracle, is patches at N = 3 either
way; marches index the same planes by code of their own.  The 64 x 64 solution
repeats across the lattice: tiles sampled at its far ends must have the bits
of a 64 x 64 run's (walls across x: of each other, away from them, and of the
run without them)."""

import numpy as np
import pytest

from paper_2306_06983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N_SIDE, TILE, STEPS = 16384, 64, 3


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    from paper_2306_06983_gb300.build import build
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("tile", [(128, 64), (64, 96)])
@pytest.mark.parametrize("wall_x", [False, True])
def test_marches(wall_x, tile):
    import torch
    from paper_2306_06983_gb300.nlbm import Simulation
    p, phi0 = W.random_smooth(TILE, TILE, 3, seed=21, model="B")
    phi0 = torch.from_numpy(np.asarray(phi0, dtype=np.float32)).cuda()
    small = Simulation(p)
    small.set_phi(phi0)
    small.step(STEPS)
    want = small.moments()
    small.close()
    reps = N_SIDE // TILE
    sim = Simulation(dict(p, nx=N_SIDE, ny=N_SIDE, wall_x=wall_x))
    sim.set_tile(*tile)
    big = phi0.repeat(1, reps, reps)
    sim.set_phi(big)
    del big
    sim.step(STEPS)
    got = sim.moments()
    sim.close()
    cols = [1, reps // 2, reps - 2] if wall_x else [0, reps // 2, reps - 1]
    for r, c in [(0, cols[0]), (reps - 1, cols[2]), (reps // 2, cols[2]), (reps - 1, cols[1])]:
        ys, xs = slice(r * TILE, (r + 1) * TILE), slice(c * TILE, (c + 1) * TILE)
        for w, g in zip(want, got):
            assert torch.equal(w, g[..., ys, xs]), (r, c)
    del sim, got
    torch.cuda.empty_cache()

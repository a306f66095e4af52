"""The step on patches against the step as a row march.

A tile with ty = 0 lets the library choose; on the small lattices here it
takes patches.  An explicit ty is a row march.  Both run the same operations
for a node, so every field of the state has the same bits."""

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


def state(p, phi0, tile):
    from paper_2306_06983_gb300.nlbm import Simulation
    sim = Simulation(p)
    if tile:
        sim.set_tile(*tile)
    sim.set_phi(phi0.astype(np.float32))
    sim.step(1)
    sim.step(4)
    out = sim.save().cpu().numpy().tobytes(), [t.cpu().numpy().tobytes() for t in sim.moments()]
    sim.close()
    return out


# Below, at and above the patch edges (16 and 32 columns, 8 rows), lattices
# smaller than a patch or its ring, odd rows, walls on every axis; the larger
# ones fill the GPU with wide patches (N <= 5, 7 and 8).
SIZES = [(1, 9, 0, 0), (3, 2, 0, 0), (15, 7, 0, 0), (16, 8, 0, 0), (17, 9, 0, 0), (33, 31, 1, 0), (4, 4, 1, 1),
         (48, 65, 0, 1), (67, 45, 1, 1), (64, 64, 0, 0), (511, 130, 0, 1), (512, 128, 0, 0)]


@pytest.mark.parametrize("nx,ny,wall_x,wall_y", SIZES)
@pytest.mark.parametrize("N,model,n", [(2, "B", 1.0), (3, "A", 1.5), (4, "B", 1.0), (5, "A", 1.0), (6, "B", 1.0),
                                       (7, "B", 1.0), (8, "A", 2.0)])
def test_patches_equal_marches(nx, ny, wall_x, wall_y, N, model, n):
    p, phi0 = W.random_smooth(nx, ny, N, seed=nx + ny, model=model, model_a_n=n, wall_x=bool(wall_x),
                              wall_y=bool(wall_y), n_disks=4)
    p = dict(p, gx=1e-6, gy=-2e-6)
    assert state(p, phi0, None) == state(p, phi0, (64, 5))


def test_patches_equal_marches_wetting_walls():
    p, phi0 = W.compound_droplet(60.0, nx=100, ny=50, R=20.0)
    p = dict(p, wall_cos=[0.3, 0.5, -0.2, 0.1])
    assert state(p, phi0, None) == state(p, phi0, (128, 7))


@pytest.mark.parametrize("N", [2, 3, 4, 5, 6, 8])
def test_ensemble_patches_equal_marches(N):
    """Members smaller than a patch, on and off its edges, of both models;
    patches of either width and marches, switched between steps (a march
    after patches needs its tile counter)."""
    from paper_2306_06983_gb300.nlbm import Batch
    mem = [W.random_smooth(nx, ny, N, seed=N + nx, model=m, wall_x=wx, wall_y=wy, n_disks=3)
           for nx, ny, m, wx, wy in ((17, 1, "B", False, False), (33, 9, "A", False, True), (64, 48, "B", False, False),
                                     (45, 30, "A", True, True), (100, 40, "B", False, True))]
    out = []
    for tiles in (((64, 5),) * 3, ((128, 0),) * 3, ((128, 8), (64, 5), (256, 8))):
        b = Batch([p for p, _ in mem])
        for k, (_, phi0) in enumerate(mem):
            b.set_phi(k, phi0.astype(np.float32))
        for tx, ty in tiles:
            b.set_tile(tx, ty)
            b.step(3)
        out.append([t.cpu().numpy().tobytes() for k in range(len(mem)) for t in b.moments(k)])
        b.close()
    assert out[0] == out[1] == out[2]

"""The result of a step does not depend on its tile: for both models at every
phase count the library's own choice (patches, one-wave marches, long marches
of narrow strips) and explicit row marches give the same bits."""

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


def state(p, phi0, tile, steps=5):
    from paper_2306_06983_gb300.nlbm import Simulation
    sim = Simulation(p)
    if tile:
        sim.set_tile(*tile)
    sim.set_phi(phi0)
    sim.step(steps)
    out = sim.save()
    sim.close()
    return out


# rows that are staged as windows and rows that are not; walls; patches of
# either width
LATTICES = [(96, 72, False, False), (67, 45, True, True), (130, 41, False, True), (512, 128, False, False)]


@pytest.mark.parametrize("model,n", [("B", 1.0), ("A", 1.0), ("A", 1.5), ("A", 3.0), ("A", 6.0)])
@pytest.mark.parametrize("N", range(2, 9))
def test_small_lattices(N, model, n):
    import torch
    for nx, ny, wall_x, wall_y in LATTICES:
        p, phi0 = W.random_smooth(nx, ny, N, seed=N, model=model, model_a_n=n, wall_x=wall_x, wall_y=wall_y, n_disks=4)
        p = dict(p, gx=1e-6, gy=-2e-6)
        phi0 = phi0.astype(np.float32)
        a = state(p, phi0, None)
        for tile in ((64, 5), (128, 40)):
            assert torch.equal(a, state(p, phi0, tile)), (nx, ny, tile)


@pytest.mark.parametrize("N,model,nx,ny", [
    (5, "B", 2048, 1472), (6, "A", 2048, 1472), (6, "B", 2048, 1472), (5, "B", 2046, 1472), (6, "B", 2046, 1472),
    (7, "A", 840, 832), (8, "B", 744, 704), (4, "B", 1116, 1088), (2, "A", 1240, 960)])
def test_marches_and_patches_at_size(N, model, nx, ny):
    """Lattices that the library marches by itself: one wave, or (N = 5 and 6,
    over 50 rows a chunk) strips of 60 columns and 20 rows; at 2046 columns
    rows are not staged as windows."""
    import torch
    p, phi0 = W.random_smooth(64, 64, N, seed=N, model=model, n_disks=4)
    phi0 = torch.from_numpy(phi0.astype(np.float32)).cuda().repeat(1, ny // 64, nx // 64 + 1)[:, :, :nx].contiguous()
    p = dict(p, nx=nx, ny=ny)
    assert torch.equal(state(p, phi0, None, 3), state(p, phi0, (128, 37), 3))

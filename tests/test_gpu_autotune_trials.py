"""The shapes that nlbm_autotune times, counted by their launches (one untimed
step and the timed ones each)."""

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


# The library's own choice is patches, one shape for every width.  400^2: the
# one-wave march has chunks of fewer than 8 rows.  2048^2: its chunks are long,
# one more trial a width.  40 columns: one width.  16-bit storage: one shape.
@pytest.mark.parametrize("nx,ny,storage,trials", [(400, 400, "f32", 1 + 3 * 7), (2048, 2048, "f32", 1 + 3 * 8),
                                                  (40, 40, "f32", 1 + 7), (512, 512, "bf16", 1)])
def test_trials(nx, ny, storage, trials):
    import torch
    from paper_2306_06983_gb300.nlbm import Simulation
    p, tile = W.random_smooth(40, 40, 3, seed=2, model="B", n_disks=3)
    p = dict(p, nx=nx, ny=ny, storage=storage)
    phi0 = torch.from_numpy(tile.astype(np.float32)).cuda().repeat(1, ny // 40 + 1, nx // 40 + 1)[:, :ny, :nx]
    a, b = Simulation(p), Simulation(p)
    for s in (a, b):
        s.set_phi(phi0)
        s.step(2)
    before = b.kernel_launches
    tx, ty, ms = b.autotune(2)
    assert b.kernel_launches - before == 3 * trials
    assert b.get_tile() == (tx, ty) and ms > 0
    a.step(3)
    b.step(3)
    assert torch.equal(a.save(), b.save())
    a.close()
    b.close()

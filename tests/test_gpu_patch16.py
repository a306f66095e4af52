"""16-bit storage on patches of either width: a periodic field repeated often
enough to fill the GPU takes wide patches (N = 5, 7 and 8), a single copy of it
narrow ones, and every copy has the bits of the single one."""

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


@pytest.mark.parametrize("storage", ["bf16", "f16"])
@pytest.mark.parametrize("N,model", [(2, "B"), (3, "A"), (4, "B"), (5, "A"), (5, "B"), (6, "A"), (7, "B"), (8, "A"), (8, "B")])
def test_copies_equal_the_single_field(N, model, storage):
    import torch
    from paper_2306_06983_gb300.nlbm import Simulation
    nx, ny, rx, ry = 90, 44, 7, 8   # 630 x 352: 880 patches of 32 x 8
    p, phi0 = W.random_smooth(nx, ny, N, seed=N, model=model, n_disks=4)
    p = dict(p, storage=storage, gx=1e-6, gy=-2e-6)
    phi0 = torch.from_numpy(phi0.astype(np.float32)).cuda()
    out = []
    for kx, ky in ((1, 1), (rx, ry)):
        sim = Simulation(dict(p, nx=nx * kx, ny=ny * ky))
        sim.set_phi(phi0.repeat(1, ky, kx).contiguous())
        sim.step(6)
        out.append(sim.moments())
        sim.close()
    for single, copies in zip(*out):
        reps = (1,) * (single.dim() - 2) + (ry, rx)
        assert torch.equal(single.repeat(*reps), copies)

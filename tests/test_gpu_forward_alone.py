"""Forwards of a gradient handle that no reverse sweep follows: after three of
them no tapes are kept, with the same bits in what they and later sweeps give."""

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


@pytest.mark.parametrize("nsteps,every", [(1, 1), (7, 1), (7, 2), (7, 3), (6, 3), (7, 7), (7, 50)])
@pytest.mark.parametrize("model,wall_y", [("A", False), ("B", True)])
def test_handle(nsteps, every, model, wall_y):
    """f forward, b sweep.  The first three forwards after a sweep, or of the
    handle, tape their last segment: the sweep need not rebuild it and has
    fewer launches."""
    import torch
    from paper_2306_06983_gb300.nlbm import AdjointRun
    p, phi0 = W.random_smooth(70, 45, 4, seed=5, model=model, wall_y=wall_y, n_disks=3)
    p["unit_delta"] = 1e-3
    phi0 = torch.from_numpy(phi0.astype(np.float32)).cuda()
    torch.cuda.synchronize()
    last = nsteps - (-(-nsteps // every) - 1) * every
    ref = None
    with torch.cuda.stream(torch.cuda.Stream()):
        run = AdjointRun(p, nsteps, every)
        alone, held = 0, False   # forwards since a sweep; whether the last segment's tapes are there
        for c in "fbffffbfbbbfffbfffffbbfb":
            before = run.kernel_launches
            if c == "f":
                phi_T = run.forward(phi0)
                assert run.kernel_launches - before == nsteps + 2
                alone, held = alone + 1, alone < 3
                ref_T = phi_T if ref is None else ref[0]
                assert torch.equal(phi_T, ref_T)
            else:
                g = run.backward(phi_T - 0.25)
                assert run.kernel_launches - before == 4 + 3 * nsteps - (last if held else 0)
                alone, held = 0, nsteps <= every   # the sweep ends with the first segment's
                ref = ref or (phi_T, *g)
                assert torch.equal(g[0], ref[1]) and np.array_equal(g[1], ref[2]) and g[2] == ref[3]
        assert run.uses_graph
        run.close()

"""The gradient run's device workspace holds what its kernels use and no more:
the checkpoints, a segment's states and tapes and the adjoint fields."""

import pytest

from paper_2306_06983_gb300 import workloads as W


@pytest.mark.parametrize("N", [2, 3, 8])
@pytest.mark.parametrize("nsteps,every", [(1, 1), (20, 5), (7, 50)])
def test_adjoint_workspace_bytes(N, nsteps, every):
    from paper_2306_06983_gb300.build import build
    from paper_2306_06983_gb300.nlbm import nlbm_adjoint_workspace_bytes
    build()
    nx, ny = 512, 384
    p, _ = W.random_smooth(64, 48, N, seed=1, model="B", n_disks=2)
    states = -(-nsteps // every) + min(every, nsteps) + 1
    floats = states * (10 * (N - 1) + 12) + min(every, nsteps) * (8 * (N - 1) + 12) + 39 * (N - 1) + 50
    got = nlbm_adjoint_workspace_bytes(dict(p, nx=nx, ny=ny), nsteps, every)
    # and the FP64 sums of the parameter gradient: one value a tile of 32 x 8
    # nodes and 256 partial sums for each
    sums = 8 * (N * (N - 1) // 2 + 1) * (nx // 32 * (ny // 8) + 256 + 1)
    assert 4 * floats * nx * ny + sums <= got <= 4 * floats * nx * ny + sums + 8 * 256

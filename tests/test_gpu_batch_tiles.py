"""The ensemble's own choice of tiles: patches for small members, marches of
32 rows where members are large; the same bits either way."""

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


@pytest.mark.parametrize("N,model,sizes,march", [
    (5, "B", [(2048, 2048)] * 2, True), (2, "A", [(2560, 2560)], True), (8, "B", [(1536, 1536)], False),
    (5, "A", [(1536, 1536)], False), (3, "B", [(2045, 1021)], False), (3, "B", [(512, 256), (64, 64), (16, 8)], False),
    (5, "B", [(2048, 2048), (1792, 2048), (60, 9)], True)])
def test_own_choice(N, model, sizes, march):
    import torch
    from paper_2306_06983_gb300.nlbm import Batch
    p, tile = W.random_smooth(64, 64, N, seed=N, model=model, n_disks=4)
    tile = torch.from_numpy(tile.astype(np.float32)).cuda()
    out = []
    for shape in (None, (256, 8), (128, 32)):
        b = Batch([dict(p, nx=nx, ny=ny) for nx, ny in sizes])
        for k, (nx, ny) in enumerate(sizes):
            b.set_phi(k, tile.repeat(1, ny // 64 + 1, nx // 64 + 1)[:, :ny, :nx].contiguous())
        if shape:
            b.set_tile(*shape)
        else:
            own = b.get_tile()
        b.step(4)
        out.append([t for k in range(len(sizes)) for t in b.moments(k)])
        torch.cuda.synchronize()
        b.close()
    px, rows = (124, 32) if march else (32, 8)
    assert own == (128, 0, sum(-(-nx // px) * -(-ny // rows) for nx, ny in sizes))
    for other in out[1:]:
        assert all(torch.equal(a, c) for a, c in zip(out[0], other))

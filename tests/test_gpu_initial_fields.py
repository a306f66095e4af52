"""Where the caller's initial phase fields may lie.  The kernel of the initial
state reads them in place where it can; memory that it cannot read so (host
memory, an odd address) and memory of the handle's own workspace, which it
writes, are copied first.  All give the state of an ordinary device array."""

import numpy as np
import pytest

from paper_2306_06983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NX, NY, N = 48, 40, 3


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    from paper_2306_06983_gb300.build import build
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build()
    torch.cuda.set_device(0)


def source(where, phi0, workspace):
    """(address, keeper) of a copy of phi0."""
    import torch
    raw = torch.from_numpy(phi0).reshape(-1).view(torch.uint8)
    if where == "pinned":
        t = raw.pin_memory()
        return t.data_ptr(), t
    if where == "odd":
        t = torch.zeros(raw.numel() + 1, dtype=torch.uint8, device="cuda")
        t[1:] = raw.cuda()
        return t.data_ptr() + 1, t
    # 4 KB into the workspace: population planes
    at = (workspace.data_ptr() + 255) // 256 * 256 + 4096 - workspace.data_ptr()
    workspace[at:at + raw.numel()] = raw.cuda()
    return workspace.data_ptr() + at, workspace


@pytest.mark.parametrize("where", ["pinned", "odd", "workspace"])
@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_simulation(where, storage):
    import torch
    from paper_2306_06983_gb300.nlbm import Simulation, nlbm_set_phi
    p, phi0 = W.random_smooth(NX, NY, N, seed=3, model="B", n_disks=3)
    p = dict(p, storage=storage)
    phi0 = phi0.astype(np.float32)
    out = []
    for kind in (None, where):
        sim = Simulation(p)
        sim.workspace.zero_()
        if kind is None:
            sim.set_phi(phi0)
        else:
            ptr, keep = source(kind, phi0, sim.workspace)
            nlbm_set_phi(sim.h, ptr)
        sim.step(3)
        out.append(sim.save())
        sim.close()
    assert torch.equal(*out)


@pytest.mark.parametrize("where", ["pinned", "odd", "workspace"])
def test_ensemble_and_gradient_run(where):
    import ctypes
    import torch
    from paper_2306_06983_gb300.nlbm import AdjointRun, Batch, nlbm_adjoint_forward, nlbm_batch_set_phi
    p, phi0 = W.random_smooth(NX, NY, N, seed=4, model="A", n_disks=3)
    phi0 = phi0.astype(np.float32)
    out = []
    for kind in (None, where):
        b, run = Batch([p, p]), AdjointRun(p, 5, 2)
        if kind is None:
            b.set_phi(0, phi0)
            b.set_phi(1, phi0)
            phi_T = run.forward(phi0)
        else:
            b.set_phi(0, phi0)
            ptr, keep = source("pinned" if kind == "workspace" else kind, phi0, None)
            nlbm_batch_set_phi(b.h, 1, ptr)
            ptr, keep2 = source(kind, phi0, run.workspace)
            phi_T = torch.empty((N, NY, NX), dtype=torch.float32, device="cuda")
            nlbm_adjoint_forward(run.h, ptr, ctypes.c_void_p(phi_T.data_ptr()))
        b.step(3)
        out.append([*b.moments(0), *b.moments(1), phi_T])
        torch.cuda.synchronize()
        b.close()
        run.close()
    assert all(torch.equal(x, y) for x, y in zip(*out))


def test_captured_into_a_graph():
    """set_phi and steps under stream capture: a replay takes the fields that
    the array holds then."""
    import torch
    from paper_2306_06983_gb300.nlbm import Simulation
    p, phi0 = W.random_smooth(NX, NY, N, seed=6, model="B", n_disks=3)
    phi0 = torch.from_numpy(phi0.astype(np.float32)).cuda()
    flipped = phi0.flip(2).contiguous()
    plain = Simulation(p)
    want = []
    for f in (phi0, flipped):
        plain.set_phi(f)
        plain.step(4)
        want.append(plain.moments())
    buf = phi0.clone()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    sim = Simulation(p, stream=stream)
    with torch.cuda.stream(stream):
        sim.set_phi(buf)   # loads the kernels
        sim.step(4)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        sim.set_phi(buf)
        sim.step(4)
    for f, w in zip((phi0, flipped), want):
        buf.copy_(f)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            got = sim.moments()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, w))
    sim.close()
    plain.close()

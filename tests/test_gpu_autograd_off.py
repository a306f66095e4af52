"""nphase_lbm where no gradient can be asked for: a plain run, without
checkpoints and tapes, of what a differentiable one takes, with the same bits."""

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


def test_nphase_lbm_without_gradients():
    import torch
    from paper_2306_06983_gb300.nlbm import NlbmError, nlbm_adjoint_workspace_bytes, nphase_lbm
    p, phi0 = W.adjoint_problem(128, 128)
    phi0 = torch.from_numpy(phi0.astype(np.float32)).cuda()
    sig, mob = torch.tensor([0.01, 0.012, 0.008], dtype=torch.float64), torch.tensor(0.1, dtype=torch.float64)
    leaf = sig.clone().requires_grad_(True)
    with_graph = nphase_lbm(phi0, leaf, mob, p, 20, 20)
    assert with_graph.requires_grad
    phi_T = with_graph.detach().clone()
    del with_graph
    full = nlbm_adjoint_workspace_bytes(dict(p, sigma=[[0, .01, .012], [.01, 0, .008], [.012, .008, 0]]), 20, 20)
    for grad, s in ((False, leaf), (True, sig)):
        torch.cuda.reset_peak_memory_stats()
        held = torch.cuda.memory_allocated()
        with torch.set_grad_enabled(grad):
            out = nphase_lbm(phi0, s, mob, p, 20, 20)
            # what a differentiable run refuses stays refused
            for bad in (dict(p, storage="bf16"), dict(p, wall_y=True, wall_cos=[0.5, 0.0, 0.0, 0.0])):
                with pytest.raises(NlbmError):
                    nphase_lbm(phi0, s, mob, bad, 20, 20)
            for steps, every in ((0, 5), (5, 0)):
                with pytest.raises(NlbmError):
                    nphase_lbm(phi0, s, mob, p, steps, every)
        assert not out.requires_grad and torch.equal(out, phi_T)
        assert torch.cuda.max_memory_allocated() - held < full / 4

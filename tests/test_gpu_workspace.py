"""Workspaces as a caller may hand them over: sub-allocated from a pool, so aligned
like the floats they hold and no further."""
import numpy as np
import pytest

import paper_2101_05888_gb300 as sas
from paper_2101_05888_gb300 import learned

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [4, 8, 12, 20])
@pytest.mark.parametrize("n", [1, 65, 500])
def test_training_workspace_at_any_float_alignment(n, offset):
    """The result does not depend on where the workspace starts, and nothing is
    written outside its sas_mlp_workspace_bytes."""
    rng = np.random.default_rng(n)
    theta = learned.init_params(3)
    frac = torch.from_numpy(rng.random(n).astype(np.float32)).cuda()
    win = torch.from_numpy((rng.standard_normal((n, 8)) + 1j * rng.standard_normal((n, 8))).astype(np.complex64)).cuda()
    tgt = torch.from_numpy((rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)).cuda()
    size = sas.sas_mlp_workspace_bytes(n)

    def run(at):
        pool = torch.full((size + 512,), 0x5A, dtype=torch.uint8, device="cuda")
        base = -pool.data_ptr() % 256                     # a 256-byte boundary of the pool
        loss, grad = torch.empty(1, device="cuda"), torch.empty(sas.SAS_MLP_NPARAMS, device="cuda")
        sas.sas_mlp_loss_grad(theta, frac, win, tgt, n, loss, grad, pool.data_ptr() + base + at)
        torch.cuda.synchronize()
        out = torch.cat([pool[:base + at], pool[base + at + size:]])
        assert bool((out == 0x5A).all())
        return loss, grad

    loss0, grad0 = run(0)
    loss1, grad1 = run(offset)
    assert torch.equal(loss0, loss1) and torch.equal(grad0, grad1)

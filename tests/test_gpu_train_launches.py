"""The training gradient where its launches change: more residual vectors than one launch
takes, and parameters that do not start on a 16-byte boundary (loss to 1e-5 and the whole
gradient to 1e-3 of the oracle's, as in test_gpu_mlp.py)."""
import numpy as np
import pytest

import cgproblems as gen
from helpers import to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2608_09647_gb300 as cg  # noqa: E402


def test_training_gradient_in_chunks_and_with_unaligned_parameters():
    """More residual vectors than one launch takes give the gradient of their mean (against the
    oracle, tolerances of test_gpu_mlp.py's whole-gradient check), and parameters that do not
    start on a 16-byte boundary give the same bits."""
    from oracle import fsai
    A = gen.q1aniso(9, 1.5, 0.7, 0.05, 2)
    h = cg.cg_create(A.n, *to_device(A))
    rng = np.random.default_rng(4)
    params = fsai.init_params(3)
    params[-65:] = rng.normal(0, 0.1, 65)
    R = rng.normal(size=(1030, A.n))
    pd = torch.from_numpy(params).cuda()
    grad = torch.empty_like(pd)
    st, loss = cg.cg_fsai_loss_grad(h, pd, grad, torch.from_numpy(R).cuda(), 0.1)
    assert st == cg.CG_OK
    Lr, gr = fsai.loss_and_grad(A, params.astype(np.float64), R, 0.1)
    assert abs(loss - Lr) <= 1e-5 * abs(Lr)
    assert np.linalg.norm(grad.cpu().numpy() - gr) <= 1e-3 * np.linalg.norm(gr)
    shifted_pd = torch.empty(pd.numel() + 1, dtype=torch.float32, device="cuda")[1:]
    shifted_pd.copy_(pd)
    g2 = torch.empty_like(grad)
    st, loss2 = cg.cg_fsai_loss_grad(h, shifted_pd, g2, torch.from_numpy(R).cuda(), 0.1)
    assert st == cg.CG_OK and loss2 == loss and torch.equal(g2, grad)
    cg.cg_destroy(h)

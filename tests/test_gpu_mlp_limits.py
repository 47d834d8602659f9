"""Training loss beyond the FP32 range, and the network's batch storage after a batch that does not fit."""
import ctypes

import pytest

from paper_2306_01085_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _batch(p=1, batch=5, hidden=64, rank=4):
    import torch
    from paper_2306_01085_gb300 import build as B
    from paper_2306_01085_gb300.dg import Mesh
    B.build()
    m = Mesh(W.box_desc(p=p, n=3))
    n = 5 * m.n_p
    m.mlp_init(hidden=hidden, rank=rank, max_samples=0, seed=5)
    g = torch.Generator(device="cuda").manual_seed(2)
    X = torch.randn(batch, n + 6, generator=g, device="cuda")
    Bs = torch.randn(batch, n, n, generator=g, device="cuda")
    return m, n, rank, X, Bs


@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("scale", [1.0, 1e15, 1e20, 1e30])
def test_loss_is_summed_in_fp64(p, scale):
    """Residual entries whose squares leave the FP32 range: the loss of FP32 residuals, summed in FP64, to 1e-6
    of the FP64 loss (see test_gpu_mlp_sizes.py)."""
    import torch
    m, n, r, X, Bs = _batch(p=p)
    Bs = Bs * scale
    prm = m.mlp_params().double()
    loss, _ = m.mlp_loss_grad(X, Bs)
    m.close()
    H, I, O = 64, n + 6, n + 2 * n * r
    parts = torch.split(prm, [H * I, H, H * H, H, O * H, O])
    h = torch.nn.functional.silu(X.double() @ parts[0].view(H, I).T + parts[1])
    h = torch.nn.functional.silu(h @ parts[2].view(H, H).T + parts[3])
    o = h @ parts[4].view(O, H).T + parts[5]
    U, V = o[:, n:n + n * r].reshape(-1, n, r), o[:, n + n * r:].reshape(-1, n, r)
    R = Bs.double() @ (torch.diag_embed(1.0 + o[:, :n]) + U @ V.transpose(1, 2)) - torch.eye(n, device="cuda")
    ref = float(R.square().sum() / (X.shape[0] * n))
    assert abs(loss - ref) <= 1e-6 * ref


def test_a_batch_that_does_not_fit_leaves_the_network_usable():
    """2^31 - 1 samples (550 GB for the first layer alone) are refused with DG_ENOMEM; the next batch is computed
    as before, and the refused allocation is not reported by its launches."""
    import torch
    from paper_2306_01085_gb300 import dg
    m, n, r, X, Bs = _batch()
    loss, grad = m.mlp_loss_grad(X, Bs)
    out = ctypes.c_double()
    rc = dg.lib().dg_mlp_loss_grad(m._h, ctypes.c_void_p(X.data_ptr()), ctypes.c_void_p(Bs.data_ptr()), 2 ** 31 - 1,
                                   ctypes.byref(out), None, None)
    assert rc == -3, rc
    again, grad2 = m.mlp_loss_grad(X, Bs)
    m.close()
    assert again == loss and torch.equal(grad, grad2)

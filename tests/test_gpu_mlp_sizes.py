"""Loss and gradients of the learned preconditioner's training batch at the edges of its tiles."""
import pytest

from paper_2306_01085_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,rank,hidden,batch", [(1, 1, 17, 1), (1, 4, 64, 65), (2, 16, 256, 70), (2, 5, 33, 3),
                                                 (2, 32, 64, 9), (3, 16, 64, 5), (3, 32, 40, 2)])
def test_loss_and_gradients_against_fp64_autograd(p, rank, hidden, batch):
    """Every gradient against FP64 autograd of the same loss, to 2e-5 in the 2-norm: FP32 sums of up to
    n_out = n (1 + 2 rank) products lose at most sqrt(n_out) 2^-24 = 9e-6 of their size. The loss to
    1e-6. Two evaluations agree bit for bit (split sums are added in a fixed order)."""
    import torch
    from paper_2306_01085_gb300 import build as B
    from paper_2306_01085_gb300.dg import Mesh
    B.build()
    m = Mesh(W.box_desc(p=p, n=3))
    n = 5 * m.n_p
    n_in, n_out = n + 6, n + 2 * n * rank
    m.mlp_init(hidden=hidden, rank=rank, max_samples=0, seed=5)
    g = torch.Generator(device="cuda").manual_seed(11)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda")
    parts = [normal(hidden, n_in) / n_in ** 0.5, 0.1 * normal(hidden), normal(hidden, hidden) / hidden ** 0.5,
             0.1 * normal(hidden), 0.3 * normal(n_out, hidden) / hidden ** 0.5, 0.05 * normal(n_out)]
    m.mlp_params(new=torch.cat([x.reshape(-1) for x in parts]))
    X = normal(batch, n_in)
    Bs = (normal(batch, n, n) * (0.5 / n ** 0.5) + torch.eye(n, device="cuda")).contiguous()
    loss, grad = m.mlp_loss_grad(X, Bs)
    again, grad2 = m.mlp_loss_grad(X, Bs)
    m.close()
    assert loss == again and torch.equal(grad, grad2)
    q = [x.double().requires_grad_(True) for x in parts]
    h = torch.nn.functional.silu(X.double() @ q[0].T + q[1])
    h = torch.nn.functional.silu(h @ q[2].T + q[3])
    o = h @ q[4].T + q[5]
    U, V = o[:, n:n + n * rank].reshape(batch, n, rank), o[:, n + n * rank:].reshape(batch, n, rank)
    R = Bs.double() @ (torch.diag_embed(1.0 + o[:, :n]) + U @ V.transpose(1, 2)) - torch.eye(n, device="cuda")
    ref = R.square().sum() / (batch * n)
    ref.backward()
    assert abs(loss - float(ref)) <= 1e-6 * float(ref)
    off = 0
    for x in q:
        got = grad[off:off + x.numel()].double()
        off += x.numel()
        err = (got - x.grad.reshape(-1)).norm() / x.grad.norm()
        assert float(err) <= 2e-5, (tuple(x.shape), float(err))

"""FP32 J v with and without the residual: the kernels that leave the value plane out do the same arithmetic."""
import pytest

from paper_2306_01085_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("n,nr", [(1, 1), (1, 3), (3, 2)])
def test_jvp_f32_without_residual_is_the_same(p, n, nr):
    """6, 18 and 108 elements: whole CTAs of 16, 8, 4, 2 and 1 elements and remainders, walls and outflow. The
    tangent is compared bit by bit (one layer of degree 2 is too coarse for the state: NaN on either side); a
    tiny, a subnormal and a zero entry of v take the conversion's other path."""
    import torch
    from paper_2306_01085_gb300 import build as B
    from paper_2306_01085_gb300.dg import Mesh
    B.build()
    d = W.shell_desc(n=n, nr=nr, p=p, euv=True)
    d.h_first = 0.0
    m = Mesh(d)
    u = torch.from_numpy(W.state_for(d, m.nodes().cpu().numpy(), 4)).cuda()
    v = torch.from_numpy(W.normal(5, u.numel()).reshape(u.shape)).cuda()
    v.view(-1)[:3] = torch.tensor([1e-40, 5e-324, 0.0], dtype=torch.float64)
    r = m.empty()
    with_r = m.jvp_f32(u, v, 0.3, r_out=r)
    assert torch.allclose(m.jvp_f32(u, v, 0.3), with_r, rtol=0.0, atol=0.0, equal_nan=True)
    m.close()

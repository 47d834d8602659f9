"""The stage operator M - c J_r for step sizes too small for M / c."""
import pytest

from paper_2306_01085_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c", [1e-150, 1e-199, 1e-201, 1e-305, 1e-309, 0.0])
@pytest.mark.parametrize("p", [1, 2])
def test_a_vanishing_step_leaves_the_mass_matrix(c, p):
    """|c J_r| is below half a unit of every entry of M: the blocks are those of c = 0 to one FP32 rounding, and the
    reduced basis over M, built with J_G w = M w, is M itself up to rounding (1e-10: 1e-16 times the condition of M)."""
    import torch
    from paper_2306_01085_gb300 import build as B
    from paper_2306_01085_gb300.dg import Mesh
    B.build()
    d = W.shell_desc(n=2, nr=3, p=p, euv=True)
    d.h_first = 0.0
    m = Mesh(d)
    u = torch.from_numpy(W.state_for(d, m.nodes().cpu().numpy(), 4)).cuda()
    b, b0 = m.block_assemble(u, 0.2, c).double(), m.block_assemble(u, 0.2, 0.0).double()
    assert bool(((b - b0).abs() <= 2.0 ** -23 * b0.abs() + 1e-13 * b0.abs().max()).all())
    w = torch.stack([torch.from_numpy(W.normal(7 + k, u.numel()).reshape(u.shape)).cuda() for k in range(3)])
    m.rb_load(w, u, 0.2, c, base="rb")
    x = torch.from_numpy(W.normal(3, u.numel()).reshape(u.shape)).cuda()
    y, ref = m.precond_apply("rb", x), m.mass_inverse(x)
    assert float((y - ref).abs().max()) <= 1e-10 * float(ref.abs().max())
    m.close()

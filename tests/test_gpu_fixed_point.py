"""The FP64 path's fixed-point contractions: range check, FP64 twin and scaling."""
import numpy as np
import pytest

from oracle import dg as OD
from oracle import mesh as OM
from paper_2306_01085_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    from paper_2306_01085_gb300 import build as B
    B.build()
    return torch


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_gradient_is_exact_under_powers_of_two_up_to_the_fp64_twin(torch_cuda, p):
    """q is linear on a periodic box, so scaling u by 2^k scales q by 2^k exactly while the exponents
    stay in the fixed-point range, and to FP64 rounding once they leave it (2^-900, 2^900: the FP64
    twin). A zero variable has a zero gradient."""
    torch = torch_cuda
    from paper_2306_01085_gb300.dg import Mesh
    m = Mesh(W.box_desc(p=p, n=3))
    u = torch.from_numpy(W.normal(3, m.n_dof).reshape(m.u_shape)).cuda()
    u[:, 2] = 0.0
    q = m.gradient(u)
    assert bool((q[:, :, 2] == 0).all())
    for k in (-300, -7, 5, 300):
        assert torch.equal(m.gradient(u * 2.0 ** k), q * 2.0 ** k), k
    for k in (-900, 900):
        err = (m.gradient(u * 2.0 ** k) * 2.0 ** -k - q).abs().max() / q.abs().max()
        assert float(err) < 1e-13, (k, float(err))
    m.close()


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_nodes_stay_in_their_neighbourhood(torch_cuda, p, bad):
    """A NaN or infinite velocity node makes its element's residual non-finite as in FP64 arithmetic,
    and leaves the elements outside its stencil bit for bit as they were."""
    torch = torch_cuda
    from paper_2306_01085_gb300.dg import Mesh
    d = W.box_desc(p=p, n=5, bc_lo=W.BC_WALL, bc_hi=W.BC_OUTFLOW, visc_exp=0.69, re=30.0)
    om = OM.OracleMesh(d)
    u = W.state_for(d, om.X, 4)
    m = Mesh(d, nodes=om.X)
    ref = m.residual(torch.from_numpy(u).cuda()).cpu().numpy()
    e = 62
    u[e, 1, 1] = bad
    r = m.residual(torch.from_numpy(u).cuda()).cpu().numpy()
    m.close()
    assert not np.isfinite(r[e]).all()
    near = om.neighbours(np.array([e]))
    near = np.union1d(np.union1d(near, om.neighbours(near)), [e])
    far = np.setdiff1d(np.arange(om.n_elem), near)
    assert np.array_equal(r[far], ref[far])


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_range_check_hands_an_element_to_the_fp64_twin(torch_cuda, p):
    """One element with a tiny momentum (2^-900) next to ordinary ones: its volume and gradient run in
    the FP64 twin and agree with the oracle like the others (1e-12 per variable)."""
    torch = torch_cuda
    from paper_2306_01085_gb300.dg import Mesh
    d = W.box_desc(p=p, n=3, bc_lo=W.BC_WALL, bc_hi=W.BC_OUTFLOW, visc_exp=0.69, re=30.0)
    om = OM.OracleMesh(d)
    u = W.state_for(d, om.X, 6)
    u[13, 2] = 2.0 ** -900
    v = W.unit_vector(9, u.shape)
    r_ref, jv_ref = OD.residual(om, u), OD.jvp(om, u, v)
    m = Mesh(d, nodes=om.X)
    r = torch.empty(m.u_shape, dtype=torch.float64, device="cuda")
    jv = m.jvp(torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(), r_out=r).cpu().numpy()
    r = r.cpu().numpy()
    m.close()
    for got, want in ((r, r_ref), (jv, jv_ref)):
        err = np.abs(got - want).max(axis=(0, 2)) / np.abs(want).max(axis=(0, 2))
        assert np.all(err <= 1e-12), err


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_mass_products_scale_exactly_and_invert(torch_cuda, p):
    """M v and M^-1 v on a shell (an odd number of elements): exact under powers of two inside the
    fixed-point range, equal to FP64 rounding outside it (the FP64 twin), a NaN node confined to its
    element, and M^-1 M v = v to 1e-12 of the largest entry."""
    torch = torch_cuda
    from paper_2306_01085_gb300.dg import Mesh
    m = Mesh(W.shell_desc(n=1, nr=7, p=p))
    v = torch.from_numpy(W.normal(8, m.n_dof).reshape(m.u_shape)).cuda()
    v[3, 1] = 0.0
    for op in (m.mass, m.mass_inverse):
        ref = op(v)
        for k in (-200, 9, 200):
            assert torch.equal(op(v * 2.0 ** k), ref * 2.0 ** k), k
        far = op(v * 2.0 ** 900) * 2.0 ** -900
        assert float(((far - ref).abs().amax((1, 2)) / ref.abs().amax((1, 2))).max()) < 1e-13
        w = v.clone()
        w[5, 2, 0] = float("nan")
        got = op(w)
        assert bool(torch.isnan(got[5, 2]).all())
        keep = torch.arange(m.n_elem, device="cuda") != 5
        assert torch.equal(got[keep], ref[keep])
    back = m.mass_inverse(m.mass(v))
    assert float((back - v).abs().max() / v.abs().max()) < 1e-12
    alias = m.mass(v)
    m.mass_inverse(alias, out=alias)
    assert torch.equal(alias, back)
    m.close()

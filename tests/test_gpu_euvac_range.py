"""EUVAC band sums over the whole range of optical depths (fixed-point sums and their FP64 fallback)."""
import numpy as np
import pytest

from oracle import dg as OD
from oracle import mesh as OM
from paper_2306_01085_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("composition", [False, True])
@pytest.mark.parametrize("scale", [1e-18, 1e-6, 1.0, 1e2, 1e4, 1e7, 1e12])
def test_heating_at_any_optical_depth(scale, composition):
    """The absorber column scaled from transparent (every attenuation rounds to 1) through depths of
    thousands (every band underflows) to arguments the fixed-point range check refuses; the flux is
    scaled back so that the heating stays visible in the energy residual. Against the oracle to 1e-12
    per variable, residual and exact Jv."""
    import torch
    from paper_2306_01085_gb300 import build as B
    from paper_2306_01085_gb300.dg import Mesh
    B.build()
    d = W.shell_desc(n=2, nr=3, p=2, euvac=True, day=172.0, composition=composition)
    d.h_first = 0.0
    d.ref_rho0 *= scale          # optical depth per reference density (the flow does not use ref_rho0)
    om = OM.OracleMesh(d)
    u = W.shell_state(om.X, d, 4)
    v = W.unit_vector(3, u.shape)
    r_ref, jv_ref = OD.residual(om, u, t=0.3), OD.jvp(om, u, v, t=0.3)
    m = Mesh(d, nodes=om.X)
    r = torch.empty(m.u_shape, dtype=torch.float64, device="cuda")
    jv = m.jvp(torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(), t=0.3, r_out=r).cpu().numpy()
    r = r.cpu().numpy()
    m.close()
    for got, want in ((r, r_ref), (jv, jv_ref)):
        err = np.abs(got - want).max(axis=(0, 2)) / np.abs(want).max(axis=(0, 2))
        assert np.all(err <= 1e-12), (scale, err)

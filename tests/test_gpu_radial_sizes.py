"""Radial implicit steps on columns shorter and longer than the LU's window of 35 and 53 unknowns."""
import numpy as np
import pytest

from oracle import radial as OR
from paper_2306_01085_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n_elem", [(1, 3), (1, 5), (1, 9), (2, 4), (2, 5), (2, 9)])
def test_step_matches_oracle(p, n_elem):
    """18 to 81 unknowns a column, two columns with different parameters: the stage solutions of the ensemble's
    Newton iteration and of the oracle's dense one agree to the Newton tolerance (1e-12 of the initial residual,
    1e-8 of the step's change as in the 28-element case)."""
    torch = pytest.importorskip("torch")
    from paper_2306_01085_gb300 import build as B
    from paper_2306_01085_gb300.dg import Radial
    B.build()
    d = W.radial_desc(n_col=2, n_elem=n_elem, p=p)
    params, u = W.radial_params(2, seed=12), W.radial_state(d, seed=13)
    dt = 30.0 / W.shell_reference().t0
    mesh, coeffs = OR.RadialMesh(d, W.radial_nodes(d)), OR.Coeffs(d)
    ref = np.stack([OR.implicit_step(mesh, u[..., c], 0.0, dt, coeffs, params[c], stages=2, tol=1e-12)[0]
                    for c in range(2)], axis=-1)
    rad = Radial(d, params, node_r=W.radial_nodes(d))
    ug = torch.from_numpy(u).cuda()
    rad.step(ug, 0.0, dt, stages=2, newton_rtol=1e-12, max_newton=30)
    got = ug.cpu().numpy()
    rad.close()
    change = np.abs(ref - u).max(axis=(0, 1, 2))
    assert np.all(change > 1e-6)
    assert np.all(np.abs(got - ref).max(axis=(0, 1, 2)) <= 1e-8 * change)

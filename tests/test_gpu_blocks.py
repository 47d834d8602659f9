"""Block-diagonal assembly of the stage operator on the GPU."""
import pytest

from paper_2306_01085_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_fp32_assembled_blocks_do_not_depend_on_the_caches():
    """Every CTA of the block-diagonal gradient reads the end-point rows from shared memory after it
    loaded them: with the operator evicted from L2 before each build, mixed-precision steps from one
    state on fresh meshes succeed and agree bit for bit."""
    import torch
    from paper_2306_01085_gb300 import build as B
    from paper_2306_01085_gb300.dg import Mesh
    B.build()
    d = W.shell_desc(n=12, nr=8, p=2, euv=True)
    evict = torch.empty(1 << 25, dtype=torch.float64, device="cuda")
    u0 = None
    seen = []
    for k in range(3):
        m = Mesh(d)
        if u0 is None:
            u0 = torch.from_numpy(W.state_for(d, m.nodes().cpu().numpy(), 4)).cuda()
        u = u0.clone()
        evict.fill_(float(k))
        st = m.implicit_step(u, 0.0, 10.0 / W.shell_reference().t0, stages=2, precond="bj16", jv_prec="f32")
        seen.append((st["gmres"], u))
        m.close()
    assert all(g == seen[0][0] and torch.equal(u, seen[0][1]) for g, u in seen)


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("composition", [False, True])
def test_blocks_are_columns_of_the_stage_operator(p, composition):
    """On a shell of three layers, wall below, outflow above (6 x 1 x 1 elements a layer; more with
    variable composition, whose profiles are undefined below the shell, where the middle of a large flat face
    lies) the block of an element, multiplied with a vector supported on it, is the element's own part of the exact FP64 stage
    operator M v - c J v; with c = 0 it is the mass matrix. FP32 storage: 2^-24 per entry, sums of n = 5 Np
    products, so n 2^-24 of max |B| |v|."""
    import torch
    from paper_2306_01085_gb300 import build as B
    from paper_2306_01085_gb300.dg import Mesh
    B.build()
    d = W.shell_desc(n=1 if not composition else 16 if p == 1 else 4, nr=3, p=p, euvac=True, day=172.0, composition=composition)
    d.h_first = 0.0
    m = Mesh(d)
    u = torch.from_numpy(W.state_for(d, m.nodes().cpu().numpy(), 4)).cuda()
    n = 5 * m.n_p
    for c in (0.7, 0.0):
        blocks = m.block_assemble(u, 0.2, c).double()
        for e in (0, 1, 2, 10):
            v = torch.zeros(m.u_shape, dtype=torch.float64, device="cuda")
            v[e] = torch.from_numpy(W.normal(5 + e, n).reshape(5, -1)).cuda()
            ref = (m.mass(v) - c * m.jvp(u, v, 0.2))[e].reshape(-1)
            got = blocks[e] @ v[e].reshape(-1)
            scale = float((blocks[e].abs() @ v[e].reshape(-1).abs()).max())
            assert float((got - ref).abs().max()) <= n * 2.0 ** -24 * scale, (c, e)
    m.close()


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_block_jacobi_applies_the_inverse_blocks(p):
    """y = B^{-1} x of block Jacobi against FP64 solves with the same assembled blocks, whose storage offsets
    take every remainder modulo 16 bytes (18 elements; n = 40 to 625 rows, up to two per thread). Gauss-Jordan
    in FP32: forward error 8 n u |B^{-1}| |B| |B^{-1}| (Higham 2002, Sec. 14.4), u = 2^-24."""
    import numpy as np
    import torch
    from paper_2306_01085_gb300 import build as B
    from paper_2306_01085_gb300.dg import Mesh
    B.build()
    d = W.shell_desc(n=1, nr=3, p=p)
    d.h_first = 0.0
    m = Mesh(d)
    u = torch.from_numpy(W.state_for(d, m.nodes().cpu().numpy(), 4)).cuda()
    n, c = 5 * m.n_p, 1e-4
    blocks = m.block_assemble(u, 0.2, c).double().cpu().numpy()
    m.precond_setup("bj", u, 0.2, c)
    x = W.normal(3, u.numel()).reshape(m.n_elem, n)
    y = m.precond_apply("bj", torch.from_numpy(x.reshape(m.u_shape)).cuda()).cpu().numpy().reshape(m.n_elem, n)
    for e in range(m.n_elem):
        inv = np.linalg.inv(blocks[e])
        bound = 8 * n * 2.0 ** -24 * (abs(inv) @ (abs(blocks[e]) @ (abs(inv) @ abs(x[e])))).max()
        assert np.abs(y[e] - inv @ x[e]).max() <= bound, e
    m.close()

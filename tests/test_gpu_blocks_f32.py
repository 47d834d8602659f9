"""FP32 assembly of the diagonal blocks (steps with an FP32 inner operator), and assemblies in several batches."""
import numpy as np
import pytest

from paper_2306_01085_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _setup(p, composition=False, **kw):
    import torch
    from paper_2306_01085_gb300 import build as B
    from paper_2306_01085_gb300.dg import Mesh
    B.build()
    d = W.shell_desc(p=p, euvac=True, day=172.0, composition=composition, **kw)
    d.h_first = 0.0
    m = Mesh(d)
    return torch, m, torch.from_numpy(W.state_for(d, m.nodes().cpu().numpy(), 4)).cuda()


@pytest.mark.parametrize("p,composition", [(1, False), (2, False), (3, False), (4, False), (2, True)])
def test_fp32_blocks_invert_the_fp64_blocks(p, composition):
    """x = B z with the FP64-assembled block B of an element (wall below, interior, outflow above) and the inverses y of
    the FP32-assembled block and y64 of the FP64-assembled one, both formed by the same FP32 elimination:
    max |y - z| <= 4 max |y64 - z| + max |B^-1 e|_abs. e bounds the assembly's error on z by that of the FP32 Jv, whose
    arithmetic it repeats column by column: per variable the largest |J_32 z - J_64 z| of the element, times c, and
    n u |M| |z|, u = 2^-24."""
    torch, m, u = _setup(p, composition, n=4 if composition else 2, nr=3)
    n, dt = 5 * m.n_p, 2.0 / W.shell_reference().t0
    t = 0.2 + dt                                        # the stage's time
    z = W.normal(9, u.numel()).reshape(m.n_elem, n)
    picked = [0, 1, m.n_elem // 2, m.n_elem - 1]
    blocks = m.block_assemble(u, t, dt)[picked].double().cpu().numpy()
    mass = m.block_assemble(u, t, 0.0)[picked].double().cpu().numpy()
    x = np.zeros((m.n_elem, n))
    for k, e in enumerate(picked):
        x[e] = blocks[k] @ z[e]
    xd = torch.from_numpy(x.reshape(m.u_shape)).cuda()
    m.precond_setup("bj", u, t, dt)
    y64 = m.precond_apply("bj", xd).cpu().numpy().reshape(m.n_elem, n)
    m.implicit_step(u.clone(), 0.2, dt, stages=1, precond="bj", jv_prec="f32")   # leaves its inverses at u behind
    y = m.precond_apply("bj", xd).cpu().numpy().reshape(m.n_elem, n)
    for k, e in enumerate(picked):
        v = torch.zeros(m.u_shape, dtype=torch.float64, device="cuda")
        v[e] = torch.from_numpy(z[e].reshape(5, -1)).cuda()
        j = (m.jvp_f32(u, v, t) - m.jvp(u, v, t))[e].abs().amax(1).cpu().numpy()
        err = dt * np.repeat(j, m.n_p) + n * 2.0 ** -24 * (np.abs(mass[k]) @ np.abs(z[e]))
        bound = 4 * np.abs(y64[e] - z[e]).max() + (np.abs(np.linalg.inv(blocks[k])) @ err).max()
        print("p", p, "e", e, "err", np.abs(y[e] - z[e]).max(), "64", np.abs(y64[e] - z[e]).max(), "bound", bound)
        assert np.abs(y[e] - z[e]).max() <= bound, e
    m.close()


def test_fp32_assembly_is_the_shorter_one():
    """The set-up of a mixed step assembles in FP32 arithmetic: beside the same inversion it takes less than 0.8 of the
    FP64 set-up (measured 0.32 with 98,304 elements)."""
    torch, m, u = _setup(2, n=16, nr=4)
    dt, ms = 2.0 / W.shell_reference().t0, {}
    for prec in ("f64", "f32"):
        ms[prec] = min(m.implicit_step(u.clone(), 0.2, dt, stages=1, precond="bj", jv_prec=prec)["precond_ms"]
                       for _ in range(4))
    m.close()
    assert ms["f32"] <= 0.8 * ms["f64"], ms


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_elements_beyond_the_first_batch(prec):
    """49,152 elements of degree 1: the Jacobians of 23,967 fill the storage in FP64 (three batches), of 47,934 in FP32
    (two). The elements at the batches' edges have the blocks of the stage operator: FP64 n 2^-24 of max |B| |v| as
    in test_gpu_blocks.py; FP32 as above, with |B| in place of |M|."""
    torch, m, u = _setup(1, n=32, nr=8)
    n, dt = 5 * m.n_p, 2.0 / W.shell_reference().t0
    picked = [0, 23966, 23967, 47933, 47934, 49151]
    c, t = dt, 0.2 + dt
    blocks = m.block_assemble(u, t, c)[picked].double()
    z = torch.from_numpy(W.normal(9, len(picked) * n).reshape(-1, n)).cuda()
    jv = {}
    for k, e in enumerate(picked):
        v = torch.zeros(m.u_shape, dtype=torch.float64, device="cuda")
        v[e] = z[k].reshape(5, -1)
        jv[e] = (m.mass(v)[e].reshape(-1), m.jvp(u, v, t)[e].reshape(-1), m.jvp_f32(u, v, t)[e].reshape(-1))
    got = torch.einsum("kij,kj->ki", blocks, z)
    if prec == "f64":
        for k, e in enumerate(picked):
            scale = float((blocks[k].abs() @ z[k].abs()).max())
            assert float((got[k] - (jv[e][0] - c * jv[e][1])).abs().max()) <= n * 2.0 ** -24 * scale, e
    else:
        x = torch.zeros(m.u_shape, dtype=torch.float64, device="cuda")
        x[picked] = got.reshape(-1, 5, m.n_p)
        m.precond_setup("bj", u, t, c)
        y64 = m.precond_apply("bj", x)[picked].reshape(-1, n)
        m.implicit_step(u.clone(), 0.2, dt, stages=1, precond="bj", jv_prec="f32")
        y = m.precond_apply("bj", x)[picked].reshape(-1, n)
        for k, e in enumerate(picked):
            d = (jv[e][2] - jv[e][1]).abs().reshape(5, -1).amax(1)
            err = c * d.repeat_interleave(m.n_p) + n * 2.0 ** -24 * (blocks[k].abs() @ z[k].abs())
            bound = 4 * float((y64[k] - z[k]).abs().max()) + float((torch.linalg.inv(blocks[k]).abs() @ err).max())
            assert float((y[k] - z[k]).abs().max()) <= bound, e
    m.close()

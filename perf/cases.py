"""The work that users of this library have it do, as measurable cases.

A case is one call (or one short sequence of calls) through the public Python entry points of
paper_2306_01085_gb300.dg: residual, gradient, exact Jacobian-vector products, block assembly and
implicit steps on boxes and cubed-sphere shells, the radial ensemble, and a training batch of the
learned preconditioner. Meshes, states and parameters are made here from the seed; sizes and options
are those of the repository's workloads, tests and benchmark, and odd sizes between them.

exact() evaluates the same discrete operators (the LDG form of Sec. 3.1 of the paper) in plain FP64
torch, with forward-mode automatic differentiation for the Jacobian-vector products.
"""
import math
import os

import numpy as np
import torch

from paper_2306_01085_gb300 import dg
from paper_2306_01085_gb300 import workloads as W

TIME = 0.37          # nondimensional time of every evaluation: the Sun away from the initial meridian


def listed():
    return [
        # the parity workload: a 4 x 4 x 4 periodic box, a few microseconds of work behind four launches
        {"name": "box4_p2_jvp", "op": "jvp", "kind": "box", "p": 2, "n": 4, "nz": 4, "walls": False, "heat": "none"},
        # the benchmarked step: fused FP64 residual and exact Jv on the 12,288-element shell
        {"name": "shell16x8_p4_jvp", "op": "jvp", "kind": "shell", "p": 4, "n": 16, "nz": 8, "heat": "none"},
        # the same call with the full physics: variable composition, eddy transport, four-absorber EUVAC
        {"name": "shell24x8_p2_comp_jvp", "op": "jvp", "kind": "shell", "p": 2, "n": 24, "nz": 8, "heat": "comp"},
        # the Newton residual of an implicit step, cubic elements, odd sizes, sub-solar heating
        {"name": "shell21x9_p3_residual", "op": "residual", "kind": "shell", "p": 3, "n": 21, "nz": 9, "heat": "gauss"},
        # the LDG gradient alone (diagnostics: vorticity, heat flux), odd sizes
        {"name": "shell13x7_p3_gradient", "op": "gradient", "kind": "shell", "p": 3, "n": 13, "nz": 7, "heat": "none"},
        # the inner operator of the mixed-precision Krylov solve
        {"name": "shell24x8_p3_jvp_f32", "op": "jvp_f32", "kind": "shell", "p": 3, "n": 24, "nz": 8, "heat": "gauss"},
        # exact diagonal blocks of the stage operator: what block-Jacobi factors and the network learns from
        {"name": "shell8x8_p2_blocks", "op": "blocks", "kind": "shell", "p": 2, "n": 8, "nz": 8, "heat": "gauss"},
        # a whole DIRK(2,2) step with the paper's own solver set-up, 10 s: reduced basis over the mass matrix, FP32 Jv
        {"name": "shell16x8_p2_step_rb", "op": "step", "kind": "shell", "p": 2, "n": 16, "nz": 8, "heat": "gauss",
         "precond": "rb", "jv_prec": "f32", "stages": 2, "dt": 10.0},
        # a whole DIRK(3,3) step of the plain FP64 solver with exact block-Jacobi, 30 s, build and solve
        {"name": "shell8x6_p2_step_plain", "op": "step", "kind": "shell", "p": 2, "n": 8, "nz": 6, "heat": "gauss",
         "precond": "bj", "jv_prec": "f64", "stages": 3, "dt": 30.0},
        # the radial ensemble of the parametric study: residual and exact Jv of 16,384 columns
        {"name": "radial16384_jvp", "op": "radial_jvp", "p": 2, "n_elem": 28, "n_col": 16384},
        # one 30 s DIRK(2,2) step of the 25 (epsilon, alpha0) pairs at 99 sites
        {"name": "radial2475_step", "op": "radial_step", "p": 2, "n_elem": 28, "n_col": 2475},
        # one training batch (loss and every parameter gradient) of the learned preconditioner
        {"name": "mlp512_p2_loss_grad", "op": "mlp", "p": 2, "batch": 512, "hidden": 256, "rank": 16},
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["jvp", "jvp", "jvp", "residual", "gradient", "jvp_f32", "blocks", "step", "radial_jvp",
                     "radial_step", "mlp"])
    if op in ("jvp", "residual", "gradient", "jvp_f32"):
        p = rng.choice([1, 2, 3, 4])
        most = 1500000 // (p + 1) ** 3                       # nodes of the benchmarked shell
        if rng.random() < 0.3:
            n = _spread(rng, 3, 16)
            return {"op": op, "kind": "box", "p": p, "n": n, "nz": _spread(rng, 3, min(24, max(3, most // (n * n)))),
                    "walls": rng.random() < 0.5, "heat": "none"}
        nz = _spread(rng, 2, 16)
        n = _spread(rng, 2, max(2, int(math.sqrt(most / (6 * nz)))))
        return {"op": op, "kind": "shell", "p": p, "n": n, "nz": nz,
                "heat": rng.choice(["none", "gauss", "euvac", "comp"])}
    if op == "blocks":
        p = rng.choice([1, 2, 3])
        nz = _spread(rng, 2, 8)
        most = 50000000 // (5 * (p + 1) ** 3) ** 2
        return {"op": op, "kind": "shell", "p": p, "n": _spread(rng, 2, max(2, int(math.sqrt(most / (6 * nz))))),
                "nz": nz, "heat": rng.choice(["none", "gauss"])}
    if op == "step":
        pc, p = rng.choice(["rb", "rb", "bj", "bj16"]), rng.choice([1, 2])
        return {"op": op, "kind": "shell", "p": p, "n": _spread(rng, 4, 16 if pc == "rb" else 12 // p),
                "nz": rng.randint(6, 8), "heat": rng.choice(["none", "gauss"]), "precond": pc,
                "jv_prec": "f32" if pc == "rb" else "f64", "stages": rng.choice([2, 3]), "dt": rng.choice([5.0, 10.0])}
    if op == "radial_jvp":
        return {"op": op, "p": 2, "n_elem": rng.randint(20, 28), "n_col": _spread(rng, 25, 16384)}
    if op == "radial_step":
        return {"op": op, "p": 2, "n_elem": rng.randint(24, 28), "n_col": _spread(rng, 25, 6000)}
    return {"op": op, "p": rng.choice([1, 2]), "batch": _spread(rng, 32, 640), "hidden": rng.choice([64, 128, 256]),
            "rank": rng.choice([4, 8, 16])}


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _desc(case):
    if case["kind"] == "box":
        d = W.box_desc(p=case["p"], n=case["n"], nz=case["nz"])
        if case["walls"]:
            d = W.box_desc(p=case["p"], n=case["n"], nz=case["nz"], bc_lo=W.BC_WALL, bc_hi=W.BC_OUTFLOW, visc_exp=0.69)
        return d
    heat = case["heat"]
    return W.shell_desc(n=case["n"], nr=case["nz"], p=case["p"], euv=heat == "gauss", euvac=heat in ("euvac", "comp"),
                        day=172.0, composition=heat == "comp")


def _gll(n):
    c = np.zeros(n)
    c[n - 1] = 1.0
    inner = np.polynomial.legendre.legroots(np.polynomial.legendre.legder(c)) if n > 2 else np.array([])
    return np.concatenate([[-1.0], np.sort(np.real(inner)), [1.0]])


def _layers(r0, r1, nz, h):
    """nz layers between r0 and r1, the first of height h, growing geometrically."""
    if h <= 0 or nz == 1:
        return r0 + (r1 - r0) * np.arange(nz + 1) / nz
    lo, hi = 1e-6, 2.0
    while h * sum(hi ** k for k in range(nz)) < r1 - r0:
        hi *= 2.0
    for _ in range(200):
        q = 0.5 * (lo + hi)
        lo, hi = (q, hi) if h * sum(q ** k for k in range(nz)) < r1 - r0 else (lo, q)
    r = r0 + np.concatenate([[0.0], np.cumsum(h * q ** np.arange(nz))])
    r[-1] = r1
    return r


def _nodes(d):
    """Node coordinates [E][3][Np] (numpy) in the numbering of include/dg.h."""
    n = d.p + 1
    s = 0.5 * (1.0 + _gll(n))
    c, b, a = [x.ravel() for x in np.meshgrid(s, s, s, indexing="ij")]
    if d.kind == W.KIND_BOX:
        k, j, i = [x.ravel() for x in np.meshgrid(range(d.nz), range(d.ny), range(d.nx), indexing="ij")]
        return np.ascontiguousarray(np.stack([(i[:, None] + a) * (d.lx / d.nx), (j[:, None] + b) * (d.ly / d.ny),
                                              (k[:, None] + c) * (d.lz / d.nz)], axis=1))
    panels = [((1, 0, 0), (0, 1, 0), (0, 0, 1)), ((0, 1, 0), (-1, 0, 0), (0, 0, 1)),
              ((-1, 0, 0), (0, -1, 0), (0, 0, 1)), ((0, -1, 0), (1, 0, 0), (0, 0, 1)),
              ((0, 0, 1), (0, 1, 0), (-1, 0, 0)), ((0, 0, -1), (0, 1, 0), (1, 0, 0))]
    rl = _layers(d.r_inner, d.r_outer, d.nz, d.h_first)
    r = rl[:-1, None] + c * (rl[1:] - rl[:-1])[:, None]                              # (nz, Np)
    cell = np.arange(d.nx)
    ta = np.tan(-0.25 * math.pi + (cell[:, None] + a) * (0.5 * math.pi / d.nx))      # (nx, Np)
    tb = np.tan(-0.25 * math.pi + (cell[:, None] + b) * (0.5 * math.pi / d.nx))
    X = np.empty((6, d.nx, d.nx, d.nz, 3, n ** 3))
    for P, (e0, e1, e2) in enumerate(panels):
        for m in range(3):
            X[P, :, :, :, m] = (e0[m] + ta[None] * e1[m] + tb[:, None] * e2[m])[:, :, None]
        X[P] /= np.sqrt((X[P] ** 2).sum(-2, keepdims=True))
    X *= r[:, None]
    return X.reshape(-1, 3, n ** 3)


def _hydrostatic(r_nd, ref):
    """rho / rho0 and T / T0 of the hydrostatic Bates atmosphere at the radii r_nd (sorted, numpy)."""
    x, w = np.polynomial.legendre.leggauss(16)
    r = np.asarray(r_nd) * ref.H0
    def temp(s):
        return 1000.0 - 800.0 * np.exp(-0.02 * ((s - W.R_EARTH) / 1e3 - 100.0))
    ends = np.concatenate([[W.R_EARTH + 100e3], r])
    lo, hi = ends[:-1], ends[1:]
    s = 0.5 * (hi - lo)[:, None] * x + 0.5 * (hi + lo)[:, None]
    f = ref.m_O * W.G_SURFACE * (W.R_EARTH / s) ** 2 / (W.K_B * temp(s))
    lnp = -np.cumsum(0.5 * (hi - lo) * (f @ w))
    return np.exp(lnp) * ref.T0 / temp(r), temp(r) / ref.T0


def _modes(rs, x, kmax=3.0):
    """A smooth random field of amplitude about one at x [..., 3] (torch): eight Fourier modes."""
    f = 0.0
    for _ in range(8):
        k = rs.normal(size=3)
        k = torch.tensor(2.0 * math.pi * kmax * rs.uniform(0.2, 1.0) * k / np.linalg.norm(k), device=x.device)
        f = f + rs.uniform(-1, 1) * torch.sin(x @ k + rs.uniform(0, 2 * math.pi))
    return f / 2.5


def _box_modes(rs, x):
    """The same on the periodic unit box (whole wave numbers)."""
    f = 0.0
    for _ in range(8):
        k = torch.tensor(2.0 * math.pi * rs.randint(-2, 3, size=3), device=x.device)
        f = f + rs.uniform(-1, 1) * torch.sin(x @ k + rs.uniform(0, 2 * math.pi))
    return f / 2.5


def _mesh_inputs(case, seed):
    """Description, nodes (numpy), state u and unit direction v (torch, GPU)."""
    d = _desc(case)
    X = _nodes(d)
    rs = np.random.RandomState(seed % (1 << 31))
    xt = torch.from_numpy(X).cuda().transpose(1, 2)
    if d.kind == W.KIND_BOX:
        f = [_box_modes(rs, xt) for _ in range(5)]
        rho, T, vel = 1.0 + 0.01 * f[0], 1.0 + 0.01 * f[4], [0.01 * f[k] for k in (1, 2, 3)]
    else:
        ref = W.shell_reference()
        n = d.p + 1
        r = np.sqrt((X[:d.nz] ** 2).sum(1)).reshape(d.nz, n, n * n)[:, :, 0].ravel()   # one column's radii
        rho1, T1 = _hydrostatic(r, ref)
        shape = (d.n_elem // d.nz, d.nz, n, n * n)
        rho = torch.from_numpy(rho1).cuda().reshape(1, d.nz, n, 1).expand(shape).reshape(d.n_elem, -1)
        T = torch.from_numpy(T1).cuda().reshape(1, d.nz, n, 1).expand(shape).reshape(d.n_elem, -1)
        unit = xt / d.r_outer
        T = T * (1.0 + 0.01 * _modes(rs, unit))
        vel = [10.0 / ref.a0 * _modes(rs, unit) for _ in range(3)]
    sr = rho.sqrt()
    u = torch.stack([rho.log(), sr * vel[0], sr * vel[1], sr * vel[2], sr * T], dim=1).contiguous()
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(u.shape, generator=g, dtype=torch.float64, device="cuda")
    return d, X, u, v / v.norm()


def _radial_inputs(case, seed):
    """Description, node radii, column parameters (numpy), state and direction (torch, GPU)."""
    d = W.radial_desc(n_col=case["n_col"], n_elem=case["n_elem"], p=case["p"])
    ref = W.shell_reference()
    rs = np.random.RandomState(seed % (1 << 31))
    rl = _layers(d.r_inner, d.r_outer, d.n_elem, d.h_first)
    r = rl[:-1, None] + 0.5 * (1.0 + _gll(d.p + 1)) * (rl[1:] - rl[:-1])[:, None]
    k = np.arange(d.n_col)
    prm = np.stack([np.array(W.RADIAL_EPS)[k % 5], np.array(W.RADIAL_ALPHA0)[(k // 5) % 5],
                    np.arcsin(rs.uniform(-1, 1, d.n_col)), rs.uniform(-math.pi, math.pi, d.n_col)], axis=1)
    rho, T = _hydrostatic(r.ravel(), ref)
    s = torch.from_numpy((r.ravel() - d.r_inner) / (d.r_outer - d.r_inner)).cuda()
    m = torch.arange(1, 5, device="cuda")
    basis = torch.cat([torch.sin(math.pi * m[:, None] * s), torch.cos(math.pi * m[:, None] * s)])       # (8, nodes)
    coef = torch.from_numpy(rs.uniform(-1, 1, (2, d.n_col, 8))).cuda()
    f = torch.einsum("acm,mi->aic", coef, basis)
    f = f / f.abs().amax(1, keepdim=True)
    rho = torch.from_numpy(rho).cuda()[:, None].expand(-1, d.n_col)
    T = torch.from_numpy(T).cuda()[:, None] * (1.0 + 0.01 * f[0])
    u = torch.stack([rho.log(), rho.sqrt() * (5.0 / ref.a0) * f[1], rho.sqrt() * T])
    u = u.reshape(3, d.n_elem, d.p + 1, d.n_col).contiguous()
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(u.shape, generator=g, dtype=torch.float64, device="cuda")
    return d, r, prm, u, v / v.norm()


def _mlp_sizes(case):
    n = 5 * (case["p"] + 1) ** 3
    n_in, n_out, h = n + 6, n + 2 * n * case["rank"], case["hidden"]
    return n, n_in, n_out, h * n_in + h + h * h + h + n_out * h + n_out


def _mlp_inputs(case, seed):
    """Parameters (W1, b1, W2, b2, W3, b3), features X and scaled blocks Bs, FP32 on the GPU."""
    n, n_in, n_out, _ = _mlp_sizes(case)
    h, nb = case["hidden"], case["batch"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    def normal(*shape):
        return torch.randn(*shape, generator=g, dtype=torch.float32, device="cuda")
    parts = [normal(h, n_in) / n_in ** 0.5, 0.1 * normal(h), normal(h, h) / h ** 0.5, 0.1 * normal(h),
             0.3 * normal(n_out, h) / h ** 0.5, 0.05 * normal(n_out)]
    X = normal(nb, n_in)
    Bs = normal(nb, n, n) * (0.5 / n ** 0.5) + torch.eye(n, device="cuda") * (1.0 + 0.5 * normal(nb, 1, n).abs())
    return parts, X, Bs.contiguous()


def _dt(case):
    return case["dt"] / W.shell_reference().t0


def prepare(case, seed):
    op = case["op"]
    if op == "mlp":
        parts, X, Bs = _mlp_inputs(case, seed)
        m = dg.Mesh(W.box_desc(p=case["p"], n=3))
        m.mlp_init(hidden=case["hidden"], rank=case["rank"], max_samples=case["batch"], seed=7)
        m.mlp_params(new=torch.cat([x.reshape(-1) for x in parts]))
        return {"op": op, "mesh": m, "X": X, "Bs": Bs}
    if op.startswith("radial"):
        d, r, prm, u, v = _radial_inputs(case, seed)
        rad = dg.Radial(d, prm, node_r=r)
        return {"op": op, "mesh": rad, "u0": u, "v": v, "u": torch.empty_like(u), "r": rad.empty(), "jv": rad.empty(),
                "dt": 30.0 / W.shell_reference().t0}
    d, X, u, v = _mesh_inputs(case, seed)
    m = dg.Mesh(d, nodes=X)
    s = {"op": op, "mesh": m, "u0": u, "v": v}
    if op == "gradient":
        s["q"] = m.empty(m.q_shape)
    elif op in ("jvp", "jvp_f32", "residual"):
        s["r"], s["jv"] = m.empty(), m.empty()
    elif op == "blocks":
        s["daii"] = 0.4358665215084590 * 60.0 / W.shell_reference().t0        # DIRK(3,3) at 60 s
    else:
        s["u"], s["dt"] = torch.empty_like(u), _dt(case)
        s["opts"] = {k: case[k] for k in ("stages", "precond", "jv_prec")}
    return s


def run(s):
    op, m = s["op"], s["mesh"]
    if op == "jvp":
        return [m.jvp(s["u0"], s["v"], t=TIME, out=s["jv"], r_out=s["r"]), s["r"]]
    if op == "jvp_f32":
        return [m.jvp_f32(s["u0"], s["v"], t=TIME, out=s["jv"], r_out=s["r"]), s["r"]]
    if op == "residual":
        return m.residual(s["u0"], t=TIME, out=s["r"])
    if op == "gradient":
        return m.gradient(s["u0"], out=s["q"])
    if op == "blocks":
        return m.block_assemble(s["u0"], TIME, s["daii"])
    if op == "step":
        s["u"].copy_(s["u0"])
        m.rb_reset()
        m.implicit_step(s["u"], TIME, s["dt"], **s["opts"])
        return s["u"]
    if op == "radial_jvp":
        return [m.jvp(s["u0"], s["v"], t=TIME, out=s["jv"], r_out=s["r"]), s["r"]]
    if op == "radial_step":
        s["u"].copy_(s["u0"])
        m.step(s["u"], TIME, s["dt"])
        return s["u"]
    loss, grad = m.mlp_loss_grad(s["X"], s["Bs"])
    return [loss, grad]


def work(case):
    """Inputs read once and outputs written once; operations of the sum-factorised passes and the
    pointwise physics of one evaluation (about 330 per point and 500 per face point in FP64)."""
    op = case["op"]
    if op == "mlp":
        n, n_in, n_out, npar = _mlp_sizes(case)
        nb, h, r = case["batch"], case["hidden"], case["rank"]
        return {"bytes": 4.0 * (nb * n_in + nb * n * n + 2 * npar),
                "flops": 6.0 * nb * (n_in * h + h * h + h * n_out) + 2.0 * nb * n * n * r * 6}
    if op.startswith("radial"):
        dof = 3 * case["n_elem"] * (case["p"] + 1) * case["n_col"]
        evals, planes = (1, 2) if op == "radial_jvp" else (10, 1)
        return {"bytes": 8.0 * dof * (4 if op == "radial_jvp" else 2), "flops": float(evals * planes * dof // 3 * 700)}
    d = _desc(case)
    n = d.p + 1
    E, NP, NF, dof = d.n_elem, d.n_p, n * n, d.n_dof
    def flops(planes):
        interp = 5 * (6 * n * NP + 12 * n * NF)
        grad = 5 * (NP * (18 + 18 * n + 36) + 3 * 12 * n * NF)
        volume = NP * (330 + 5 * (6 * n + 12 + 6 * n))
        return planes * E * (interp + grad + volume + 3 * NF * 500.0)
    nodes = 24.0 * E * NP
    if op == "jvp" or op == "jvp_f32":
        return {"bytes": 32.0 * dof + nodes, "flops": flops(2)}
    if op == "residual":
        return {"bytes": 16.0 * dof + nodes, "flops": flops(1)}
    if op == "gradient":
        return {"bytes": 32.0 * dof + nodes, "flops": E * 5.0 * (6 * n * NP + 12 * n * NF + NP * (54 + 18 * n + 18 * n))}
    nb = 5 * NP
    if op == "blocks":
        return {"bytes": 4.0 * E * nb * nb + 8.0 * dof + nodes, "flops": nb * flops(1)}
    iters = case["stages"] * 3 * 12
    if case["precond"] == "rb":
        return {"bytes": (16.0 + 32.0 * iters) * dof + nodes, "flops": iters * flops(1)}
    return {"bytes": 16.0 * dof + nodes + iters * E * nb * nb * (2.0 if case["precond"] == "bj16" else 4.0),
            "flops": nb * flops(1) + iters * flops(1)}


# ------------------------------------------------------------------------------------------------
# the same operators in plain FP64 torch
# ------------------------------------------------------------------------------------------------
def _lagrange(x, t):
    return np.array([[np.prod([(ti - x[m]) / (x[k] - x[m]) for m in range(len(x)) if m != k]) for k in range(len(x))]
                     for ti in t])


def _ops1d(n):
    """GLL -> Gauss, Gauss derivative, end-point rows and weights."""
    xg, wg = np.polynomial.legendre.leggauss(n)
    B = _lagrange(_gll(n), xg)
    lam = np.array([1.0 / np.prod([xg[k] - xg[m] for m in range(n) if m != k]) for k in range(n)])
    D = np.zeros((n, n))
    for i in range(n):
        for k in range(n):
            if i != k:
                D[i, k] = lam[k] / lam[i] / (xg[i] - xg[k])
        D[i, i] = -D[i].sum()
    ends = _lagrange(xg, [-1.0, 1.0])
    t = [torch.from_numpy(a).cuda() for a in (B, D, ends, wg)]
    return t[0], t[1], t[2], t[3]


def _along(A, f, axis):
    """A applied along reference axis 0, 1 or 2 of f [..., k, j, i] (axis 0 is the last one)."""
    if axis == 0:
        return torch.einsum("qa,...kja->...kjq", A, f)
    if axis == 1:
        return torch.einsum("qa,...kai->...kqi", A, f)
    return torch.einsum("qa,...aji->...qji", A, f)


def _at_faces(ends, f):
    """Values of f [..., n, n, n] on the six faces [..., 6, n * n] (axis-major, low end first)."""
    out = []
    for axis in range(3):
        for side in range(2):
            out.append(_along(ends[side:side + 1], f, axis).reshape(*f.shape[:-3], -1))
    return torch.stack(out, dim=-2)


def _lift(ends, g, axis, side, n):
    """sum over the face of g [..., n * n] times the end-point rows: [..., n, n, n]."""
    e = ends[side]
    g = g.reshape(*g.shape[:-1], n, n)
    if axis == 0:
        return torch.einsum("...kj,i->...kji", g, e)
    if axis == 1:
        return torch.einsum("...ki,j->...kji", g, e)
    return torch.einsum("...ji,k->...kji", g, e)


class _Geometry:
    def __init__(self, d, X):
        self.d, self.n = d, d.p + 1
        n, E = self.n, X.shape[0]
        self.B, self.D, self.ends, self.w = _ops1d(n)
        X = torch.from_numpy(X).cuda()
        rel = (X - X[:, :, :1]).reshape(E, 3, n, n, n)
        xr = rel
        for a in range(3):
            xr = _along(self.B, xr, a)
        J = torch.stack([_along(self.D, xr, a) for a in range(3)], dim=2)                # [E, d, a, ...]
        self.xg = xr + X[:, :, 0].reshape(E, 3, 1, 1, 1)
        cof = torch.stack([torch.cross(J[:, :, 1], J[:, :, 2], dim=1), torch.cross(J[:, :, 2], J[:, :, 0], dim=1),
                           torch.cross(J[:, :, 0], J[:, :, 1], dim=1)], dim=1)           # [E, a, d, ...]
        wq = self.w[:, None, None] * self.w[None, :, None] * self.w[None, None, :]
        self.G = wq * cof
        self.W = wq * (J[:, :, 0] * cof[:, 0]).sum(1)
        Jf = _at_faces(self.ends, J)                                                     # [E, d, a, 6, nf]
        wf = (self.w[:, None] * self.w[None, :]).reshape(-1)
        nds = []
        for f in range(6):
            a1, a2 = (f // 2 + 1) % 3, (f // 2 + 2) % 3
            nds.append((1 if f % 2 else -1) * torch.cross(Jf[:, :, a1, f], Jf[:, :, a2, f], dim=1))
        nds = torch.stack(nds, dim=1)                                                    # [E, 6, d, nf]
        self.nds, self.area = wf * nds, wf * nds.square().sum(2).sqrt()
        self._connect(_at_faces(self.ends, xr).permute(0, 2, 1, 3) + X[:, None, :, :1], X, n)

    def _connect(self, xf, X, n):
        d, E = self.d, X.shape[0]
        self.xf = xf                                                                     # [E, 6, 3, nf]
        idx = torch.arange(n ** 3).reshape(n, n, n)
        corners = [idx[:, :, 0], idx[:, :, -1], idx[:, 0], idx[:, -1], idx[0], idx[-1]]
        cen = torch.stack([X[:, :, c[::n - 1, ::n - 1].reshape(-1).cuda()].mean(-1) for c in corners], dim=1)
        per = torch.zeros(3, dtype=torch.float64, device="cuda")
        if d.kind == W.KIND_BOX:
            per = torch.tensor([d.lx, d.ly, d.lz if d.bc_lo == W.BC_PERIODIC else 0.0], dtype=torch.float64, device="cuda")
        key = cen.reshape(-1, 3).clone()
        for a in range(3):
            if per[a] > 0:
                key[:, a] = torch.remainder(key[:, a] + 1e-9, per[a])
        s = key @ torch.tensor([0.8191725134, 0.3710290461, 0.4378120987], dtype=torch.float64, device="cuda")
        order = torch.argsort(s)
        a, b = order[:-1], order[1:]
        near = (key[a] - key[b]).abs().amax(1) < 1e-9 * float(X.abs().max())
        a, b = a[near], b[near]
        other = torch.full((E * 6,), -1, dtype=torch.long, device="cuda")
        other[a], other[b] = b, a
        self.inner = torch.nonzero(other >= 0).reshape(-1)
        self.other = other[self.inner]
        x = xf.reshape(E * 6, 3, n * n)
        c = x.mean(-1, keepdim=True)
        perm = []
        for own, oth in zip(self.inner.split(20000), self.other.split(20000)):
            dist = ((x[own] - c[own]).unsqueeze(-1) - (x[oth] - c[oth]).unsqueeze(-2)).square().sum(1)
            perm.append(dist.argmin(-1))
        self.perm = torch.cat(perm)                                                      # the other's point
        rest = torch.nonzero(other < 0).reshape(-1)
        if d.kind == W.KIND_BOX:
            low = cen.reshape(-1, 3)[rest, 2].abs() < 1e-9
        else:
            r = x[rest].square().sum(1).sqrt().mean(-1)
            low = (r - d.r_inner).abs() < (r - d.r_outer).abs()
        kind = torch.where(low, d.bc_lo, d.bc_hi)
        self.wall, self.out = rest[kind == W.BC_WALL], rest[kind == W.BC_OUTFLOW]

    def across(self, t):
        """The neighbour's values of t [E * 6, ..., nf] on the interior faces, in the own point order."""
        p = self.perm.reshape(self.perm.shape[0], *([1] * (t.dim() - 2)), -1).expand(-1, *t.shape[1:-1], -1)
        return torch.gather(t[self.other], -1, p)


def _mixture(d, x):
    """m*, c_v*, grad c_v*, conductivity factor and mass fractions (variable composition); x [..., 3, pts]."""
    r = x.square().sum(-2).sqrt()
    inv = [1.0, 16.0 / 28.0, 16.0 / 32.0, 16.0 / 4.0]
    al = [1.0, 3.6 / 5.6, 3.6 / 5.6, 1.0]
    a, b = d.comp_a, d.comp_b
    chi = [sum(a[2 * s + j] * torch.exp(b[2 * s + j] * r) for j in range(2)) for s in range(3)]
    dchi = [sum(a[2 * s + j] * b[2 * s + j] * torch.exp(b[2 * s + j] * r) for j in range(2)) for s in range(3)]
    chi, dchi = [1.0 - chi[0] - chi[1] - chi[2]] + chi, [-(dchi[0] + dchi[1] + dchi[2])] + dchi
    cv = sum(c * i for c, i in zip(chi, inv))
    dcv = sum(c * i for c, i in zip(dchi, inv))
    kf = sum(c * i * q for c, i, q in zip(chi, inv, al)) / cv
    return 1.0 / cv, cv, [dcv * x[..., k, :] / r for k in range(3)], kf, chi


def _bands():
    """The EUVAC table of the paper's appendix: wavelength, flux, A and cross sections (N2, O2, O, He)."""
    with open(os.path.join("tests", "golden", "euvac_table.txt")) as f:
        rows = [x.split() for x in f if x.strip() and not x.startswith("#")]
    lam = [np.mean([float(y) for y in x[0].split("-")]) * 1e-10 for x in rows]
    return [(l, float(x[1]) * 1e26, float(x[2]), [float(y) for y in x[3:7]]) for l, x in zip(lam, rows)]


def _heating(d, u0, T, r, cchi, mstar, weights):
    """Nondimensional EUVAC heating (efficiency one); weights: chi_s m_O / m_s of O, N2, O2, He."""
    kB, H0 = 1.380649e-23, 1.380649e-23 * d.ref_T0 / (d.ref_m * d.ref_g0)
    a0, cv0 = math.sqrt(d.gamma * kB * d.ref_T0 / d.ref_m), kB / ((d.gamma - 1.0) * d.ref_m)
    n0 = d.ref_rho0 * torch.exp(u0) / d.ref_m
    H = H0 * T * (r / d.g_r0) ** 2 / mstar
    rt = r * H0 / H
    cchi = cchi.clamp(-1.0, 1.0)
    schi = (1.0 - cchi ** 2).clamp(min=0.0).sqrt()
    day = cchi > 0
    lit = day | (schi * r > d.g_r0)
    ex = torch.special.erfcx((rt / 2).sqrt() * cchi.abs())
    base = (math.pi * rt / 2).sqrt()
    ch = torch.where(day, base * ex, base * (2.0 * torch.exp(torch.where(day | ~lit, 0.0 * rt, rt * (1.0 - schi))) - ex))
    ch = torch.where(lit, ch, 0.0 * ch)
    q = 0.0
    fbar = 0.5 * (d.euv_f107 + d.euv_f107a)
    for lam, flux, A, (pn2, po2, po, phe) in _bands():
        I0 = flux * max(0.8, 1.0 + A * (fbar - 80.0)) / d.euv_dsun ** 2
        absorb = n0 * (weights[0] * po + weights[1] * pn2 + weights[2] * po2 + weights[3] * phe)
        q = q + absorb * I0 * torch.exp(-absorb * H * ch) * (6.62607015e-34 * 299792458.0 / lam)
    return torch.where(lit, q, 0.0 * q) * H0 / (d.ref_rho0 * cv0 * d.ref_T0 * a0)


def _sun(d, t):
    w = 2.0 * math.pi / 365.24
    delta = math.asin(math.sin(-23.44 * math.pi / 180.0)
                      * math.cos(w * (d.euv_day + 9.0) + 2.0 * 0.0167 * math.sin(w * (d.euv_day - 3.0))))
    wt = d.euv_omega_t * t
    return [-math.cos(delta) * math.cos(wt), math.cos(delta) * math.sin(wt), math.sin(delta)]


class _Physics:
    """Fluxes and sources at points: u [.., 5, pts], q [.., 3, 5, pts], x [.., 3, pts]."""

    def __init__(self, d):
        self.d = d
        self.cmu, self.ck = 1.0 / math.sqrt(d.gamma * d.grashof), math.sqrt(d.gamma / d.grashof) / d.prandtl
        self.cd = (d.gamma - 1.0) * math.sqrt(d.gamma / d.grashof)

    def mix(self, x):
        d = self.d
        return _mixture(d, x) if d.comp else (d.mass, 1.0 / d.mass, None, 1.0, None)

    def transport(self, T, u0, mx):
        d = self.d
        if d.comp:
            rho = torch.exp(u0)
            return (T * mx[0]).sqrt() + d.eddy_nu * rho, mx[3] * T ** 0.69 + d.eddy_alpha * rho / mx[0]
        mu = T ** d.visc_exp if d.visc_exp else torch.ones_like(T)
        return mu, mu

    def primitives(self, u, q, mx):
        isr = torch.exp(-0.5 * u[..., 0, :])
        v = [u[..., 1 + m, :] * isr for m in range(3)]
        T = u[..., 4, :] * isr
        gv = [[isr * (q[..., k, 1 + m, :] - 0.5 * u[..., 1 + m, :] * q[..., k, 0, :]) for k in range(3)] for m in range(3)]
        gT = [isr * (q[..., k, 4, :] - 0.5 * u[..., 4, :] * q[..., k, 0, :]) for k in range(3)]
        div = gv[0][0] + gv[1][1] + gv[2][2]
        eps = [[gv[m][k] + gv[k][m] - (2.0 / 3.0 * div if m == k else 0.0) for k in range(3)] for m in range(3)]
        mu, kappa = self.transport(T, u[..., 0, :], mx)
        return isr, v, T, gv, gT, div, eps, mu, kappa

    def flux(self, u, q, x, viscous=True):
        """F [.., 5, 3, pts]."""
        mx = self.mix(x)
        isr, v, T, gv, gT, div, eps, mu, kappa = self.primitives(u, q, mx)
        pc = 1.0 / (self.d.gamma * mx[0])
        rows = [torch.stack([u[..., 0, :] * v[k] for k in range(3)], dim=-2)]
        for m in range(3):
            rows.append(torch.stack([u[..., 1 + m, :] * v[k] + (pc * u[..., 4, :] if m == k else 0.0)
                                     - (self.cmu * mu * isr * eps[m][k] if viscous else 0.0) for k in range(3)], dim=-2))
        rows.append(torch.stack([u[..., 4, :] * v[k] - (self.ck * kappa * isr / mx[1] * gT[k] if viscous else 0.0)
                                 for k in range(3)], dim=-2))
        return torch.stack(rows, dim=-3)

    def sigma(self, u, x):
        mx = self.mix(x)
        isr = torch.exp(-0.5 * u[..., 0, :])
        mu, kappa = self.transport(u[..., 4, :] * isr, u[..., 0, :], mx)
        lam = self.d.lambda0 + 0.0 * isr
        sm = lam + self.cmu * mu * isr
        return torch.stack([lam, sm, sm, sm, lam + self.ck * kappa * isr / mx[1]], dim=-2)

    def wall(self, u):
        z = 0.0 * u[..., 0, :]
        return torch.stack([u[..., 0, :], z, z, z, torch.exp(0.5 * u[..., 0, :]) * self.d.t_wall], dim=-2)

    def source(self, u, q, x, t):
        d, mx = self.d, self.mix(x)
        isr, v, T, gv, gT, div, eps, mu, kappa = self.primitives(u, q, mx)
        sr = torch.exp(0.5 * u[..., 0, :])
        r = x.square().sum(-2).sqrt()
        X = [x[..., k, :] for k in range(3)]
        g = [d.gvec[k] + 0.0 * r for k in range(3)] if d.gravity_kind == 0 else [-(d.g_r0 / r) ** 2 / r * X[k] for k in range(3)]
        def rot(y):
            w = d.omega
            return [w[1] * y[2] - w[2] * y[1], w[2] * y[0] - w[0] * y[2], w[0] * y[1] - w[1] * y[0]]
        cen, cor = rot(rot(X)), rot(v)
        acc = [g[k] / d.gamma - d.froude ** 2 / d.gamma * cen[k] - 2.0 * d.froude / math.sqrt(d.gamma) * cor[k] for k in range(3)]
        pc, u4 = 1.0 / (d.gamma * mx[0]), u[..., 4, :]
        s = [(u[..., 0, :] - 1.0) * div]
        for m in range(3):
            eg = sum(eps[m][k] * q[..., k, 0, :] for k in range(3))
            s.append(sr * acc[m] + 0.5 * div * u[..., 1 + m, :] - 0.5 * pc * u4 * q[..., m, 0, :] + 0.5 * self.cmu * mu * isr * eg)
        tg = sum(gT[k] * q[..., k, 0, :] for k in range(3))
        diss = sum(eps[m][k] * gv[m][k] for m in range(3) for k in range(3))
        ck = self.ck * kappa * isr / mx[1]
        s4 = (1.5 - d.gamma) * u4 * div + 0.5 * ck * tg + self.cd * mu * isr / mx[1] * diss
        if d.comp:
            s4 = s4 - sum((u4 * v[k] - ck * gT[k]) * mx[2][k] for k in range(3)) / mx[1]
        if d.euv == W.EUV_GAUSS:
            sx, sy = math.cos(d.euv_omega_t * t), -math.sin(d.euv_omega_t * t)
            chi = torch.arccos(((X[0] * sx + X[1] * sy) / r).clamp(-1.0, 1.0))
            heat = d.euv_amp * torch.exp(-chi ** 2 / (2 * d.euv_sigma ** 2) - math.log(2.0) * ((r - d.euv_r_peak) / d.euv_width) ** 2)
            s4 = s4 + heat * isr / mx[1]
        elif d.euv == W.EUV_EUVAC:
            sun = _sun(d, t)
            wt = [mx[4][0], mx[4][1] * 16 / 28, mx[4][2] * 16 / 32, mx[4][3] * 4.0] if d.comp else [1.0 / d.mass, 0.0, 0.0, 0.0]
            heat = _heating(d, u[..., 0, :], T, r, (X[0] * sun[0] + X[1] * sun[1] + X[2] * sun[2]) / r, mx[0], wt)
            s4 = s4 + d.euv_eff * heat * isr / mx[1]
        return torch.stack(s + [s4], dim=-2)


def _gradient(g, ph, u):
    """Gauss values of u, its traces [E * 6, 5, nf] and the LDG gradient [E, 3, 5, n, n, n] at the Gauss points."""
    n, E = g.n, u.shape[0]
    U = u.reshape(E, 5, n, n, n)
    for a in range(3):
        U = _along(g.B, U, a)
    UF = _at_faces(g.ends, U).permute(0, 2, 1, 3).reshape(E * 6, 5, n * n)
    hat = UF.clone()
    hat[g.inner] = 0.5 * (UF[g.inner] + g.across(UF))
    hat[g.wall] = ph.wall(UF[g.wall])
    hat = hat.reshape(E, 6, 5, n * n)
    q = 0.0
    for a in range(3):
        q = q - _along(g.D.T.contiguous(), g.G[:, a, :, None] * U[:, None], a)
        for side in range(2):
            f = 2 * a + side
            q = q + _lift(g.ends, g.nds[:, f, :, None] * hat[:, f, None], a, side, n)
    return U, UF, q / g.W[:, None, None]


def _residual(g, ph, u, t):
    n, E = g.n, u.shape[0]
    U, UF, Q = _gradient(g, ph, u)
    QF = _at_faces(g.ends, Q).permute(0, 3, 1, 2, 4).reshape(E * 6, 3, 5, n * n)
    pts = n ** 3
    Uv, Qv, xv = U.reshape(E, 5, pts), Q.reshape(E, 3, 5, pts), g.xg.reshape(E, 3, pts)
    F = ph.flux(Uv, Qv, xv)                                                              # [E, 5, 3, pts]
    r = (g.W.reshape(E, 1, pts) * ph.source(Uv, Qv, xv, t)).reshape(E, 5, n, n, n)
    nds, area, xf = g.nds.reshape(E * 6, 1, 3, n * n), g.area.reshape(E * 6, 1, n * n), g.xf.reshape(E * 6, 3, n * n)
    i, o, w = g.inner, g.out, g.wall
    fh = torch.zeros_like(UF)
    Fo = ph.flux(UF, QF, xf)
    u2 = g.across(UF)
    mean = 0.5 * (UF[i] + u2)
    fh[i] = (0.5 * (Fo[i] + g.across(Fo)) * nds[i]).sum(2) + ph.sigma(mean, xf[i]) * (UF[i] - mean) * area[i]
    ub = ph.wall(UF[w])
    fh[w] = (ph.flux(ub, QF[w], xf[w]) * nds[w]).sum(2) + ph.sigma(ub, xf[w]) * (UF[w] - ub) * area[w]
    fh[o] = (ph.flux(UF[o], QF[o], xf[o], viscous=False) * nds[o]).sum(2)
    fh = fh.reshape(E, 6, 5, n * n)
    for a in range(3):
        Fa = (g.G[:, a].reshape(E, 1, 3, pts) * F).sum(2).reshape(E, 5, n, n, n)
        r = r + _along(g.D.T.contiguous(), Fa, a)
        for side in range(2):
            r = r - _lift(g.ends, fh[:, 2 * a + side], a, side, n)
    for a in range(3):
        r = _along(g.B.T.contiguous(), r, a)
    return r.reshape(E, 5, pts)


def _radial_residual(d, r, prm, u, t):
    """The symmetric restriction of the same form on every column: u [3, E, n, nc] -> r."""
    n = d.p + 1
    B, D, ends, w = _ops1d(n)
    eps, alpha, lat, lon = [torch.from_numpy(np.ascontiguousarray(prm[:, k])).cuda() for k in range(4)]
    site = [lat.cos() * lon.cos(), lat.cos() * lon.sin(), lat.sin()]
    rn = torch.from_numpy(r).cuda()
    rL, rR, rg = rn[:, 0], rn[:, -1], rn @ B.T
    J = 0.5 * (rR - rL)[:, None]
    Wt, G, T2 = [x.unsqueeze(-1) for x in (w * J * rg ** 2, w * rg ** 2, 2.0 * w * J * rg)]
    rgc = rg.unsqueeze(-1)
    cmu, ckk = 1.0 / math.sqrt(d.gamma * d.grashof), math.sqrt(d.gamma / d.grashof) / d.prandtl
    cd, pc, cv = (d.gamma - 1.0) * math.sqrt(d.gamma / d.grashof), 1.0 / (d.gamma * d.mass), 1.0 / d.mass
    def prim(a, q):
        isr = torch.exp(-0.5 * a[0])
        T = a[2] * isr
        gvr, gvt, gT = isr * (q[1] - 0.5 * a[1] * q[0]), isr * q[2], isr * (q[3] - 0.5 * a[2] * q[0])
        div = gvr + 2.0 * gvt
        mu = T ** d.visc_exp
        return isr, a[1] * isr, T, gvr, gvt, gT, div, 2 * gvr - 2.0 / 3.0 * div, 2 * gvt - 2.0 / 3.0 * div, mu, alpha * mu
    def flux(a, q, viscous=True):
        isr, v, T, gvr, gvt, gT, div, er, et, mu, kap = prim(a, q)
        s = 1.0 if viscous else 0.0
        return torch.stack([a[0] * v, a[1] * v + pc * a[2] - s * cmu * mu * isr * er, a[2] * v - s * ckk * kap * isr / cv * gT])
    def sigma(a):
        isr = torch.exp(-0.5 * a[0])
        mu = (a[2] * isr) ** d.visc_exp
        return torch.stack([d.lambda0 + 0.0 * isr, d.lambda0 + cmu * mu * isr, d.lambda0 + ckk * alpha * mu * isr / cv])
    def wall(a):
        return torch.stack([a[0], 0.0 * a[0], torch.exp(0.5 * a[0]) * d.t_wall])
    U = torch.einsum("gi,ceik->cegk", B, u)
    lo, hi = u[:, :, 0], u[:, :, -1]
    hat = torch.cat([wall(lo[:, 0])[:, None], 0.5 * (hi[:, :-1] + lo[:, 1:]), hi[:, -1:]], dim=1)
    def lifted(f):
        return (torch.einsum("cek,j->cejk", f[:, 1:] * (rR ** 2)[:, None], ends[1])
                - torch.einsum("cek,j->cejk", f[:, :-1] * (rL ** 2)[:, None], ends[0]))
    q3 = (lifted(hat) - T2 * U - torch.einsum("gj,cegk->cejk", D, G * U)) / Wt
    Q = torch.stack([q3[0], q3[1], U[1] / rgc, q3[2]])
    qlo, qhi = torch.einsum("j,cejk->cek", ends[0], Q), torch.einsum("j,cejk->cek", ends[1], Q)
    mid = 0.5 * (hi[:, :-1] + lo[:, 1:])
    Fi = 0.5 * (flux(hi[:, :-1], qhi[:, :-1]) + flux(lo[:, 1:], qlo[:, 1:])) + sigma(mid) * 0.5 * (hi[:, :-1] - lo[:, 1:])
    ub = wall(lo[:, 0])
    Fb = flux(ub, qlo[:, 0]) - sigma(ub) * (lo[:, 0] - ub)
    Fh = torch.cat([Fb[:, None], Fi, flux(hi[:, -1], qhi[:, -1], False)[:, None]], dim=1)
    F = flux(U, Q)
    isr, v, T, gvr, gvt, gT, div, er, et, mu, kap = prim(U, Q)
    cm, ck = cmu * mu * isr, ckk * kap * isr / cv
    sun = _sun(d, t)
    cchi = (site[0] * sun[0] + site[1] * sun[1] + site[2] * sun[2]).expand_as(T)
    heat = eps * _heating(d, U[0], T, rgc.expand_as(T), cchi, d.mass, [1.0 / d.mass, 0.0, 0.0, 0.0])
    S = torch.stack([(U[0] - 1.0) * div,
                     torch.exp(0.5 * U[0]) * (-(d.g_r0 / rgc) ** 2 / d.gamma) + 0.5 * div * U[1] - 0.5 * pc * U[2] * Q[0]
                     + 0.5 * cm * er * Q[0] + 2.0 / rgc * (pc * U[2] - cm * et),
                     heat * isr / cv + (1.5 - d.gamma) * U[2] * div + 0.5 * ck * gT * Q[0]
                     + cd * mu * isr / cv * (er * gvr + 2.0 * et * gvt)])
    R = Wt * S + torch.einsum("gj,cegk->cejk", D, G * F) - lifted(Fh)
    return torch.einsum("gi,cegk->ceik", B, R)


def exact(case, seed):
    op = case["op"]
    if op in ("blocks", "step", "radial_step"):
        return None              # thousands of operator applications: minutes in plain torch
    if op == "mlp":
        parts, X, Bs = _mlp_inputs(case, seed)
        n, _, _, _ = _mlp_sizes(case)
        r, nb = case["rank"], case["batch"]
        p = [x.double().requires_grad_(True) for x in parts]
        h = torch.nn.functional.silu(X.double() @ p[0].T + p[1])
        h = torch.nn.functional.silu(h @ p[2].T + p[3])
        o = h @ p[4].T + p[5]
        U, V = o[:, n:n + n * r].reshape(nb, n, r), o[:, n + n * r:].reshape(nb, n, r)
        P = torch.diag_embed(1.0 + o[:, :n]) + U @ V.transpose(1, 2)
        R = Bs.double() @ P - torch.eye(n, dtype=torch.float64, device="cuda")
        loss = R.square().sum() / (nb * n)
        loss.backward()
        return [float(loss), torch.cat([x.grad.reshape(-1) for x in p])]
    if op == "radial_jvp":
        d, r, prm, u, v = _radial_inputs(case, seed)
        res, jv = torch.func.jvp(lambda a: _radial_residual(d, r, prm, a, TIME), (u,), (v,))
        return [jv, res]
    d, X, u, v = _mesh_inputs(case, seed)
    g, ph = _Geometry(d, X), _Physics(d)
    if op == "gradient":
        _, _, Q = _gradient(g, ph, u)
        Binv = torch.linalg.inv(g.B)
        for a in range(3):
            Q = _along(Binv, Q, a)
        return Q.reshape(d.n_elem, 3, 5, -1)
    if op == "residual":
        return _residual(g, ph, u, TIME)
    res, jv = torch.func.jvp(lambda a: _residual(g, ph, a, TIME), (u,), (v,))
    return [jv, res]

"""Performance cases of the matrix-free operator library: the calls that its users make, at the sizes they make them.

Each case is a dict of plain values.  `kind` names the path:

  apply    y = A x of the mass or diffusion operator (ceed_apply_mass / ceed_apply_diffusion)
  batch    several meshes of different order, several components and right-hand sides, one persistent launch
  cg       ceed_cg_solve: Jacobi-PCG in FP64, or mixed precision with reliable updates
  adjoint  diffusion_k forward and backward: A(k) x, then dL/dx and dL/dk
  tet      the non-tensor operator on tetrahedra (ceed_nt_apply)

Meshes are structured lattices of the unit cube whose interior vertices are moved by up to a tenth of the
spacing, the shapes of the bake-off problems; the coefficient is 1 + 0.5 sin sin sin unless the case says
otherwise.  Inputs come from the seed alone, the mesh's vertices included.
"""
import math

import numpy as np
import torch

import paper_2109_05072_gb300 as ceed

DEV = "cuda"
PREC = {"f64": ceed.CEED_F64, "df": ceed.CEED_F64_DF, "f32": ceed.CEED_F32}
QBYTES = {"f64": 8, "df": 8, "f32": 4}


def listed():
    return [
        # the smallest call: mass operator on 4^3 elements of degree 2, 729 nodes (a coarse level, a unit test, one
        # implicit step of a toy problem): launches and latency are all of it
        _apply("mass_p2_4cube", 4, 4, 4, 2, rule="gauss", op="mass"),
        # a small ragged mesh with Dirichlet rows, one rank's share of a larger run: too few elements to fill the chip
        _apply("diff_p5_13x11x9_masked", 13, 11, 9, 5, masked=True),
        # BP5 at p = 7, FP64, the operator this library is quoted on (22.2M nodes)
        _apply("diff_p7_40cube", 40, 40, 40, 7),
        # BP1 at p = 6: Gauss mass operator of an explicit time step, ragged lattice
        _apply("mass_p6_gauss_27x25x23", 27, 25, 23, 6, rule="gauss", op="mass"),
        # BP4: vector diffusion (3 components, 4 right-hand sides) with Gauss quadrature at low order
        _apply("diff_p3_gauss_3c4r", 21, 19, 17, 3, rule="gauss", ncomp=3, nrhs=4),
        # BP5 at p = 7 with the FP64-accurate double-float quadrature data
        _apply("diff_p7_df_32cube", 32, 32, 32, 7, prec="df"),
        # the low-precision operator of mixed-precision solvers, on the masked problem they solve
        _apply("diff_p7_f32_40cube_masked", 40, 40, 40, 7, prec="f32", masked=True),
        # orders 3, 5, 7 in one persistent launch, 3 components x 4 right-hand sides, Gauss
        dict(name="batch_p357_3c4r", kind="batch", n3=24, n5=20, n7=16, ncomp=3, nrhs=4),
        # Jacobi-PCG in FP64, a fixed number of iterations (the bake-off's CG timing)
        dict(name="cg_fp64_p7_24cube", kind="cg", nx=24, ny=24, nz=24, p=7, mode="fp64", iters=100),
        # a whole solve to 1e-10: FP32 inner operator, FP64 residuals (reliable updates)
        dict(name="cg_mixed_p7_16cube", kind="cg", nx=16, ny=16, nz=16, p=7, mode="mixed", iters=0),
        # parameter identification: forward and gradient with a lognormal coefficient per point
        dict(name="adjoint_p4_32cube", kind="adjoint", nx=32, ny=32, nz=32, p=4, stored=True, df=False),
        # degree-4 tetrahedra, FP64
        dict(name="tet_p4_24cube", kind="tet", nx=24, ny=24, nz=24, p=4),
    ]


def _apply(name, nx, ny, nz, p, rule="gll", op="diff", prec="f64", masked=False, ncomp=1, nrhs=1):
    return dict(name=name, kind="apply", nx=nx, ny=ny, nz=nz, p=p, rule=rule, op=op, prec=prec, masked=masked,
                ncomp=ncomp, nrhs=nrhs)


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lattice(rng, p, cols, most):
    """Three element counts, each side within a factor of two of the others, at most `most` node values."""
    nodes = math.exp(rng.uniform(math.log(700), math.log(most)))
    side = max(1.0, (nodes / cols) ** (1 / 3) / p)
    n = [max(1, int(round(side * 2 ** rng.uniform(-0.5, 0.5)))) for _ in range(3)]
    while (n[0] * p + 1) * (n[1] * p + 1) * (n[2] * p + 1) * cols > 1.1 * most and max(n) > 1:
        n[n.index(max(n))] -= 1
    return n


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "apply", "batch", "cg", "adjoint", "tet"])
    if kind == "apply":
        p = rng.randint(1, 8)
        prec = rng.choice(["f64", "f64", "f64", "df", "f32"])
        ncomp, nrhs = rng.choice([(1, 1), (1, 1), (1, 1), (3, 1), (1, 4), (3, 4)])
        n = _lattice(rng, p, ncomp * nrhs, 2.0e7)
        c = _apply("", *n, p, rule=rng.choice(["gll", "gll", "gauss"]),
                   op="diff" if prec == "f32" else rng.choice(["diff", "diff", "mass"]), prec=prec,
                   masked=rng.random() < 0.5, ncomp=ncomp, nrhs=nrhs)
        del c["name"]
        return c
    if kind == "batch":
        s = rng.uniform(4, 16)
        return dict(kind="batch", n3=int(1.5 * s), n5=int(1.25 * s), n7=int(s), ncomp=rng.choice([1, 3]),
                    nrhs=rng.choice([1, 2, 4]))
    if kind == "cg":
        p = rng.randint(2, 8)
        n = [_logint(rng, 20, 110) // p + 1 for _ in range(3)]
        mode = rng.choice(["fp64", "mixed"])
        return dict(kind="cg", nx=n[0], ny=n[1], nz=n[2], p=p, mode=mode, iters=rng.randint(40, 100) if mode == "fp64" else 0)
    if kind == "adjoint":
        p = rng.randint(1, 8)
        n = _lattice(rng, p, 1, 4.0e6)
        stored = rng.random() < 0.7
        return dict(kind="adjoint", nx=n[0], ny=n[1], nz=n[2], p=p, stored=stored, df=stored and rng.random() < 0.3)
    p = rng.randint(1, 4)
    n = _lattice(rng, p, 1, 9.0e5)
    return dict(kind="tet", nx=n[0], ny=n[1], nz=n[2], p=p)


# ---------------------------------------------------------------- 1D rules and bases (FP64)

def _gll(n):
    if n == 2:
        x = np.array([-1.0, 1.0])
    else:
        L = np.polynomial.legendre.Legendre.basis(n - 1)
        x = np.concatenate([[-1.0], np.sort(L.deriv().roots().real), [1.0]])
        for _ in range(3):  # Newton on the derivative: the companion matrix leaves the last few bits
            x[1:-1] -= L.deriv()(x[1:-1]) / L.deriv(2)(x[1:-1])
    P = np.polynomial.legendre.Legendre.basis(n - 1)(x)
    return x, 2.0 / (n * (n - 1) * P * P)


def _lagrange(xn, xq):
    """Values and derivatives at xq of the Lagrange basis on xn: B[q, n], D[q, n]."""
    n = len(xn)
    B, D = np.ones((len(xq), n)), np.zeros((len(xq), n))
    for j in range(n):
        den = np.prod([xn[j] - xn[m] for m in range(n) if m != j])
        B[:, j] = np.prod([xq - xn[m] for m in range(n) if m != j], axis=0) / den
        for l in range(n):
            if l != j:
                rest = [xq - xn[m] for m in range(n) if m not in (j, l)]
                D[:, j] += (np.prod(rest, axis=0) if rest else 1.0) / den
    return B, D


# ---------------------------------------------------------------- inputs, from the seed alone

def _gen(seed, tag):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + tag)
    return g


def _uniform(n, seed, tag):
    return torch.rand(n, generator=_gen(seed, tag), device=DEV, dtype=torch.float64) * 2 - 1


def _corner_lattice(nx, ny, nz, seed):
    """Vertex positions [nz+1, ny+1, nx+1, 3] of the unit cube's lattice, interior ones moved."""
    ax = [torch.arange(n + 1, device=DEV, dtype=torch.float64) / n for n in (nx, ny, nz)]
    X = torch.stack([ax[0][None, None, :].expand(nz + 1, ny + 1, nx + 1), ax[1][None, :, None].expand(nz + 1, ny + 1, nx + 1),
                     ax[2][:, None, None].expand(nz + 1, ny + 1, nx + 1)], -1).contiguous()
    off = _uniform(X.numel(), seed, 1).reshape(X.shape) * torch.tensor([0.1 / nx, 0.1 / ny, 0.1 / nz], device=DEV, dtype=torch.float64)
    X[1:-1, 1:-1, 1:-1] += off[1:-1, 1:-1, 1:-1]
    return X


def _hexes(nx, ny, nz, p, seed):
    """A hexahedral lattice: elem_dofs [E, P^3], vertices [E, 8, 3], boundary mask [n], n."""
    X = _corner_lattice(nx, ny, nz, seed)
    V = torch.stack([X[(v >> 2):(v >> 2) + nz, ((v >> 1) & 1):((v >> 1) & 1) + ny, (v & 1):(v & 1) + nx] for v in range(8)], 3)
    Mx, My, Mz = p * nx + 1, p * ny + 1, p * nz + 1
    ar = lambda n: torch.arange(n, device=DEV, dtype=torch.int64)
    base = (p * ar(nx))[None, None, :] + Mx * ((p * ar(ny))[None, :, None] + My * (p * ar(nz))[:, None, None])
    loc = ar(p + 1)[None, None, :] + Mx * (ar(p + 1)[None, :, None] + My * ar(p + 1)[:, None, None])
    dofs = (base.reshape(-1, 1) + loc.reshape(1, -1)).to(torch.int32)
    return dofs, V.reshape(-1, 8, 3).contiguous(), _boundary(Mx, My, Mz), Mx * My * Mz


def _boundary(Mx, My, Mz):
    edge = lambda n: (torch.arange(n, device=DEV) % max(1, n - 1)) == 0
    return (edge(Mz)[:, None, None] | edge(My)[None, :, None] | edge(Mx)[None, None, :]).reshape(-1).to(torch.uint8)


def _load(nx, ny, nz, p, seed):
    """A right-hand side: a smooth source (eight sine modes with random amplitudes, zero on the boundary) times the
    nodes' quadrature weights on the undisturbed lattice."""
    xn, wn = _gll(p + 1)
    amp, mode = _uniform(8, seed, 5), torch.randint(1, 5, (3, 8), generator=_gen(seed, 6), device=DEV)
    f = []
    for d, n in enumerate((nx, ny, nz)):
        e = np.arange(n)[:, None]
        at = e * p + np.arange(p + 1)
        x = np.empty(p * n + 1)
        x[at] = (e + (xn + 1) / 2) / n
        w = np.bincount(at.reshape(-1), np.tile(wn / (2 * n), n))
        x, w = torch.from_numpy(x).to(DEV), torch.from_numpy(w).to(DEV)
        s = torch.sin(math.pi * mode[d][:, None] * x) * w
        s[:, 0] = s[:, -1] = 0.0
        f.append(s)
    return torch.einsum("mz,my,mx->zyx", amp[:, None] * f[2], f[1], f[0]).reshape(-1)


PATHS = (((0, 1, 2), 1), ((0, 2, 1), -1), ((1, 0, 2), -1), ((1, 2, 0), 1), ((2, 0, 1), 1), ((2, 1, 0), -1))


def _tet_nodes(p):
    return np.array([(i, j, k) for k in range(p + 1) for j in range(p + 1 - k) for i in range(p + 1 - j - k)])


def _tets(nx, ny, nz, p, seed):
    """Every cube of the lattice split into six tetrahedra of positive volume; degree-p equispaced nodes."""
    X = _corner_lattice(nx, ny, nz, seed)
    Mx, My, Mz = p * nx + 1, p * ny + 1, p * nz + 1
    ar = lambda n: torch.arange(n, device=DEV, dtype=torch.int64)
    base = (p * ar(nx))[None, None, :] + Mx * ((p * ar(ny))[None, :, None] + My * (p * ar(nz))[:, None, None])
    verts, dofs = [], []
    for perm, sign in PATHS:
        c = np.zeros((4, 3), dtype=np.int64)
        for s, a in enumerate(perm):
            c[s + 1] = c[s]
            c[s + 1, a] += 1
        if sign < 0:
            c[[2, 3]] = c[[3, 2]]
        verts.append(torch.stack([X[z:z + nz, y:y + ny, x:x + nx] for x, y, z in c], 3))
        L = _tet_nodes(p) @ c[1:]
        dofs.append(base[..., None] + torch.from_numpy(L[:, 0] + Mx * (L[:, 1] + My * L[:, 2])).to(DEV))
    E = 6 * nx * ny * nz
    return (torch.stack(dofs, 3).reshape(E, -1).to(torch.int32), torch.stack(verts, 3).reshape(E, 4, 3).contiguous(),
            _boundary(Mx, My, Mz), Mx * My * Mz)


def _gauss_jacobi(n, alpha):
    """Points and weights on [0, 1] for the weight (1 - t)^alpha (Golub and Welsch)."""
    k = np.arange(n, dtype=np.float64)
    diag = np.full(n, -alpha / (alpha + 2.0))
    diag[1:] = -alpha ** 2 / ((2 * k[1:] + alpha) * (2 * k[1:] + alpha + 2))
    m = k[1:]
    off = 2 * m * (m + alpha) / ((2 * m + alpha) * np.sqrt((2 * m + alpha + 1) * (2 * m + alpha - 1)))
    x, V = np.linalg.eigh(np.diag(diag) + np.diag(off, 1) + np.diag(off, -1))
    return (x + 1) / 2, V[0] ** 2 / (alpha + 1)


def _tet_basis(p):
    """Equispaced Lagrange basis of degree p on the reference tetrahedron, conical product rule of p + 1 points."""
    (tu, wu), (tv, wv), (ts, ws) = (_gauss_jacobi(p + 1, a) for a in (2, 1, 0))
    u, v, s = (a.reshape(-1) for a in np.meshgrid(tu, tv, ts, indexing="ij"))
    W = (wu[:, None, None] * wv[None, :, None] * ws[None, None, :]).reshape(-1)
    xi = np.stack([u, (1 - u) * v, (1 - u) * (1 - v) * s], -1)
    mi = _tet_nodes(p)
    mono = lambda X: np.stack([X[:, 0] ** i * X[:, 1] ** j * X[:, 2] ** k for i, j, k in mi], -1)
    C = np.linalg.inv(mono(mi / p))
    grad = []
    for d in range(3):
        m = mi.copy()
        m[:, d] = np.maximum(m[:, d] - 1, 0)
        G = np.stack([mi[n, d] * xi[:, 0] ** m[n, 0] * xi[:, 1] ** m[n, 1] * xi[:, 2] ** m[n, 2] for n in range(len(mi))], -1)
        grad.append(G @ C)
    return mono(xi) @ C, np.stack(grad), W, xi


# ---------------------------------------------------------------- prepare and run

def _qrule(case):
    return ceed.CEED_QRULE_GAUSS if case.get("rule") == "gauss" else ceed.CEED_QRULE_GLL


def _batch_parts(case):
    return [(case["n%d" % p], p) for p in (3, 5, 7)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _prepare_batch(case, seed)
    if kind == "tet":
        return _prepare_tet(case, seed)
    dofs, verts, bnd, n = _hexes(case["nx"], case["ny"], case["nz"], case["p"], seed)
    if kind == "adjoint":
        m = ceed.ceed_setup_mesh(dofs.shape[0], n, case["p"], dofs, verts, bnd)
        geo = None
        if case["stored"]:
            geo = ceed.alloc_qdata(m, ceed.CEED_OP_DIFFUSION, ceed.CEED_F64)
            ceed.ceed_build_geometry(m, geo)
        k = _lognormal(m.n_elem * m.nq, seed).reshape(m.n_elem, m.nq)
        return dict(case=case, mesh=m, geo=geo, k=k.requires_grad_(), x=_uniform(n, seed, 2).requires_grad_(), g=_uniform(n, seed, 3))
    if kind == "cg":
        m = ceed.ceed_setup_mesh(dofs.shape[0], n, case["p"], dofs, verts, bnd)
        op = ceed.CEED_OP_DIFFUSION
        qd = _qdata(m, op, ceed.CEED_F64)
        st = dict(case=case, mesh=m, qdata=qd, b=_load(case["nx"], case["ny"], case["nz"], case["p"], seed), x=torch.empty(n, device=DEV, dtype=torch.float64))
        if case["mode"] == "mixed":
            st["opts"] = dict(mode=ceed.CEED_CG_MIXED_RELIABLE, op=op, tol=1e-10, qdata_lo=_qdata(m, op, ceed.CEED_F32), prec_lo=ceed.CEED_F32)
        else:
            st["opts"] = dict(mode=ceed.CEED_CG_FP64, op=op, fixed_iters=case["iters"])
        st["work"] = torch.empty(ceed.ceed_cg_workspace_bytes(m, **st["opts"]), dtype=torch.uint8, device=DEV)
        return st
    op = ceed.CEED_OP_MASS if case["op"] == "mass" else ceed.CEED_OP_DIFFUSION
    prec = PREC[case["prec"]]
    m = ceed.ceed_setup_mesh(dofs.shape[0], n, case["p"], dofs, verts, bnd, q_rule=_qrule(case), ncomp=case["ncomp"])
    qd = _qdata(m, op, prec)
    x = _uniform(n * case["ncomp"] * case["nrhs"], seed, 2)
    y = torch.empty_like(x)
    if case["prec"] == "f32":
        # the brick kernel where the lattice has bricks, as measured; its sums at shared nodes are in an order of
        # their own, so a program that wants the same bits on every run fixes the variant
        if ceed.ceed_mesh_bricks(m) and x.numel() == n:
            ceed.ceed_set_apply_variant(m, op, prec, 1, 2)
    else:
        ceed.ceed_autotune_apply(m, op, qd, prec, x, y, case["nrhs"])
    return dict(case=case, mesh=m, qdata=qd, prec=prec, x=x, y=y,
                apply=ceed.ceed_apply_mass if case["op"] == "mass" else ceed.ceed_apply_diffusion,
                flags=ceed.CEED_APPLY_DIRICHLET if case["masked"] else 0)


def _qdata(m, op, prec):
    qd = ceed.alloc_qdata(m, op, prec)
    ceed.ceed_build_qdata(m, op, ceed.CEED_COEFF_SINE, None, prec, qd)
    return qd


def _lognormal(n, seed):
    return torch.exp(0.5 * torch.randn(n, generator=_gen(seed, 4), device=DEV, dtype=torch.float64))


def _prepare_batch(case, seed):
    ms, qs, xs, ys = [], [], [], []
    for n1, p in _batch_parts(case):
        dofs, verts, bnd, n = _hexes(n1, n1, n1, p, seed + p)
        m = ceed.ceed_setup_mesh(dofs.shape[0], n, p, dofs, verts, bnd, q_rule=ceed.CEED_QRULE_GAUSS, ncomp=case["ncomp"])
        ms.append(m)
        qs.append(_qdata(m, ceed.CEED_OP_DIFFUSION, ceed.CEED_F64))
        xs.append(_uniform(n * case["ncomp"] * case["nrhs"], seed + p, 2))
        ys.append(torch.empty_like(xs[-1]))
    b = ceed.ceed_batch_create(ms, qs, ceed.CEED_F64, ceed.CEED_OP_DIFFUSION, xs, ys, case["nrhs"])
    ceed.ceed_batch_autotune(b)
    return dict(case=case, batch=b, ys=ys)


def _prepare_tet(case, seed):
    dofs, verts, bnd, n = _tets(case["nx"], case["ny"], case["nz"], case["p"], seed)
    h = ceed.ceed_nt_setup(dofs.shape[0], n, *_tet_basis(case["p"]), dofs, verts, bnd)
    qd = ceed.alloc_nt_qdata(h, ceed.CEED_OP_DIFFUSION, ceed.CEED_F64)
    ceed.ceed_nt_build_qdata(h, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, ceed.CEED_F64, qd)
    x = _uniform(n, seed, 2)
    return dict(case=case, nt=h, qdata=qd, x=x, y=torch.empty_like(x))


def run(state):
    case = state["case"]
    if case["kind"] == "apply":
        state["apply"](state["mesh"], state["qdata"], state["prec"], state["x"], state["y"], case["nrhs"], state["flags"])
        return state["y"]
    if case["kind"] == "batch":
        ceed.ceed_batch_apply(state["batch"])
        return state["ys"]
    if case["kind"] == "cg":
        ceed.ceed_cg_solve(state["mesh"], state["qdata"], ceed.CEED_F64, state["b"], state["x"], work=state["work"], **state["opts"])
        return state["x"]
    if case["kind"] == "adjoint":
        y = ceed.diffusion_k(state["x"], state["k"], state["mesh"], state["geo"], case["df"])
        gx, gk = torch.autograd.grad(y, (state["x"], state["k"]), state["g"])
        return dict(y=y.detach(), gx=gx, gk=gk)
    ceed.ceed_nt_apply(state["nt"], ceed.CEED_OP_DIFFUSION, state["qdata"], ceed.CEED_F64, state["x"], state["y"])
    return state["y"]


# ---------------------------------------------------------------- what a pass cannot do without

def _hex_work(E, p, Q, op, cols, n, qbytes):
    """One application: every node value read and written once, the quadrature data and the element map read once;
    the multiplications and additions of the sum-factorized passes and of the pointwise step."""
    P, nq = p + 1, Q ** 3
    bytes_ = 16.0 * n * cols + E * (nq * qbytes * (1 if op == "mass" else 6) + 4.0 * P ** 3)
    interp = 0 if Q == P else 2 * 2 * (P ** 3 * Q + P ** 2 * Q ** 2 + P * Q ** 3)
    flops = E * cols * (interp + (nq if op == "mass" else 12.0 * Q ** 4 + 15.0 * nq))
    return bytes_, flops


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        for n1, p in _batch_parts(case):
            bb, ff = _hex_work(n1 ** 3, p, p + 2, "diff", case["ncomp"] * case["nrhs"], (p * n1 + 1) ** 3, 8)
            b, f = b + bb, f + ff
        return dict(bytes=b, flops=f)
    p = case["p"]
    E = case["nx"] * case["ny"] * case["nz"]
    n = (p * case["nx"] + 1) * (p * case["ny"] + 1) * (p * case["nz"] + 1)
    if kind == "apply":
        b, f = _hex_work(E, p, p + 2 if case["rule"] == "gauss" else p + 1, case["op"], case["ncomp"] * case["nrhs"], n, QBYTES[case["prec"]])
    elif kind == "cg":
        # one iteration: the operator, and eleven passes over vectors (p.q read with the operator's; x, r, z and p
        # updated).  A solve to a tolerance takes about 33 iterations per element along a side at p = 7
        mixed = case["mode"] == "mixed"
        it = case["iters"] or 4.8 * p * max(case["nx"], case["ny"], case["nz"])
        b, f = _hex_work(E, p, p + 1, "diff", 1, n, 4 if mixed else 8)
        b, f = it * (b + 72.0 * n), it * (f + 12.0 * n)
    elif kind == "adjoint":
        P3 = (p + 1) ** 3
        geo = 48.0 * P3 if case["stored"] else 192.0
        b = 40.0 * n + E * (2 * geo + 24.0 * P3 + 8.0 * P3)
        f = E * (12.0 * (p + 1) ** 4 + 21.0 * P3 + 18.0 * (p + 1) ** 4 + 36.0 * P3)
    else:
        P, Q = (p + 1) * (p + 2) * (p + 3) // 6, (p + 1) ** 3
        E *= 6
        b, f = 16.0 * n + E * (48.0 * Q + 4.0 * P), E * (12.0 * P * Q + 15.0 * Q)
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------- the same in plain torch, 64 bits

def _t3(c, b, a, u):
    """v[e, k, j, i] = sum c[k, z] b[j, y] a[i, x] u[e, z, y, x], one direction at a time (u may have more axes at its end)."""
    u = torch.einsum("ix,ezyx...->ezyi...", a, u)
    u = torch.einsum("jy,ezyi...->ezji...", b, u)
    return torch.einsum("kz,ezji...->ekji...", c, u)


class _Hex:
    """The operator on a hexahedral lattice by definition: einsums over element arrays, index_add to the nodes."""

    def __init__(self, dofs, verts, bnd, n, p, rule, k="sine"):
        P = p + 1
        xn, wn = _gll(P)
        xq, wq = (xn, wn) if rule == "gll" else np.polynomial.legendre.leggauss(P + 1)
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
        B, D = _lagrange(xn, xq)
        self.B, self.D = t(B), t(D)
        self.dofs, self.n, self.P, self.Q, self.bnd = dofs.long(), n, P, len(xq), bnd
        h, dh = np.stack([(1 - xq) / 2, (1 + xq) / 2], -1), np.array([[-0.5, 0.5]] * len(xq))
        V = verts.reshape(-1, 2, 2, 2, 3)  # [e, vz, vy, vx, c]
        ev = lambda a, b, c: _t3(t(c), t(b), t(a), V)
        X, J = ev(h, h, h), torch.stack([ev(dh, h, h), ev(h, dh, h), ev(h, h, dh)], -1)  # J[..., c, d]
        w = t(wq)
        w = w[:, None, None] * w[None, :, None] * w[None, None, :]
        det = torch.linalg.det(J)
        if k == "sine":
            k = 1 + 0.5 * torch.sin(2 * math.pi * X).prod(-1)
        self.mass = w * det * k
        adj = torch.linalg.inv(J) * det[..., None, None]  # rows: reference directions
        self.Ghat = (w / det)[..., None, None] * (adj @ adj.transpose(-1, -2))
        self.k = k

    def grad(self, x):
        u = x[self.dofs].reshape(-1, self.P, self.P, self.P)
        B, D = self.B, self.D
        return torch.stack([_t3(B, B, D, u), _t3(B, D, B, u), _t3(D, B, B, u)], -1)

    def grad_t(self, v):
        B, D = self.B.T, self.D.T
        return self.scatter(_t3(B, B, D, v[..., 0]) + _t3(B, D, B, v[..., 1]) + _t3(D, B, B, v[..., 2]))

    def scatter(self, ye):
        return torch.zeros(self.n, device=DEV, dtype=torch.float64).index_add_(0, self.dofs.reshape(-1), ye.reshape(-1))

    def diffusion(self, x, k):
        return self.grad_t(torch.einsum("ekjiab,ekjib->ekjia", self.Ghat * k[..., None, None], self.grad(x)))

    def apply(self, op, x, masked=False):
        x0 = torch.where(self.bnd != 0, 0.0, x) if masked else x
        if op == "mass":
            B = self.B
            u = _t3(B, B, B, x0[self.dofs].reshape(-1, self.P, self.P, self.P))
            y = self.scatter(_t3(B.T, B.T, B.T, self.mass * u))
        else:
            y = self.diffusion(x0, self.k)
        return torch.where(self.bnd != 0, x, y) if masked else y

    def diagonal(self):
        B, D = self.B, self.D
        G = self.Ghat * self.k[..., None, None]
        f = [(B, B, D), (B, D, B), (D, B, B)]
        d = 0
        for a in range(3):
            for b in range(3):
                m = [f[a][s] * f[b][s] for s in range(3)]
                d = d + _t3(*(f.T for f in m), G[..., a, b])
        return torch.where(self.bnd != 0, 1.0, self.scatter(d))


def _exact_apply(h, case, x):
    cols = case["ncomp"] * case["nrhs"]
    xs = x.reshape(h.n, cols)
    return torch.stack([h.apply(case["op"], xs[:, c].contiguous(), case["masked"]) for c in range(cols)], -1).reshape(-1)


def _exact_cg(h, b, iters):
    d = h.diagonal()
    x, r = torch.zeros_like(b), b.clone()
    z = r / d
    p, rz, stop = z.clone(), torch.dot(r, z), 1e-13 * torch.linalg.norm(b)
    for it in range(iters or 5000):
        q = h.apply("diff", p, True)
        a = rz / torch.dot(p, q)
        x += a * p
        r -= a * q
        if not iters and it % 20 == 19 and torch.linalg.norm(r) < stop:
            break
        z = r / d
        rz, old = torch.dot(r, z), rz
        p = z + (rz / old) * p
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for n1, p in _batch_parts(case):
            dofs, verts, bnd, n = _hexes(n1, n1, n1, p, seed + p)
            h = _Hex(dofs, verts, bnd, n, p, "gauss")
            out.append(_exact_apply(h, dict(case, op="diff", masked=False), _uniform(n * case["ncomp"] * case["nrhs"], seed + p, 2)))
        return out
    if kind == "tet":
        return _exact_tet(case, seed)
    dofs, verts, bnd, n = _hexes(case["nx"], case["ny"], case["nz"], case["p"], seed)
    if kind == "adjoint":
        Q = case["p"] + 1
        k = _lognormal(dofs.shape[0] * Q ** 3, seed).reshape(-1, Q, Q, Q)
        h = _Hex(dofs, verts, bnd, n, case["p"], "gll", k)
        x, g = _uniform(n, seed, 2), _uniform(n, seed, 3)
        gk = torch.einsum("ekjia,ekjiab,ekjib->ekji", h.grad(g), h.Ghat, h.grad(x)).reshape(-1, Q ** 3)
        return dict(y=h.diffusion(x, k), gx=h.diffusion(g, k), gk=gk)
    h = _Hex(dofs, verts, bnd, n, case["p"], case.get("rule", "gll"))
    if kind == "cg":
        return _exact_cg(h, _load(case["nx"], case["ny"], case["nz"], case["p"], seed), case["iters"])
    return _exact_apply(h, case, _uniform(n * case["ncomp"] * case["nrhs"], seed, 2))


def _exact_tet(case, seed):
    dofs, verts, _, n = _tets(case["nx"], case["ny"], case["nz"], case["p"], seed)
    _, grad, w, xi = (torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in _tet_basis(case["p"]))
    x, y = _uniform(n, seed, 2), torch.zeros(n, device=DEV, dtype=torch.float64)
    for a in range(0, dofs.shape[0], 20000):
        d, V = dofs[a:a + 20000].long(), verts[a:a + 20000]
        J = (V[:, 1:] - V[:, :1]).transpose(1, 2)  # J[c, d]
        det = torch.linalg.det(J)
        adj = torch.linalg.inv(J) * det[:, None, None]
        X = V[:, None, 0] + torch.einsum("ecd,qd->eqc", J, xi)
        k = 1 + 0.5 * torch.sin(2 * math.pi * X).prod(-1)
        G = (adj @ adj.transpose(1, 2)) / det[:, None, None]
        u = torch.einsum("dqn,en->eqd", grad, x[d])
        v = torch.einsum("eab,eqb->eqa", G, u) * (k * w)[..., None]
        y.index_add_(0, d.reshape(-1), torch.einsum("dqn,eqd->en", grad, v).reshape(-1))
    return y

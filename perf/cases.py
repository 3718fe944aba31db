"""The framework's work on space-time HDG trace systems, as cases to be timed.

A user assembles a trace system on the GPU, builds an l-AIR hierarchy of it, applies the V-cycle inside a
Krylov method, and, in an optimisation loop, solves the adjoint system and asks for the gradient with respect
to the element velocities.  Each case is one of these calls (or one whole step) on the Kuhn meshes that the
repository's tests and benchmark use: [0,1]^2 (1D + time) or [0,1]^3 (2D + time), n cubes per direction,
degree p.  The flow, the data and the right-hand sides come from the seed; the mesh and the reference tables
are a user's constants.

Keys of a case: op; D, n, p (space-time dimension, cubes per direction, degree); nu; noise (standard deviation of
the element velocities); prec (0 FP64, 1 FP32, 2 BF16 off-diagonals); block (facet blocks in the finest
operator); falgout (0: the first pass of Ruge-Stueben, else the block length of the blocked splitting);
distance; relax; theta, theta_r; rtol; k and dtype of the many right-hand-side V-cycle.
"""
import functools
import math

import numpy as np
import torch

import paper_2010_11130_gb300 as air
from paper_2010_11130_gb300 import hdg
from sthdg.mesh import build_mesh, choose_reflection

PI = math.pi
DEV = "cuda"
DIRICHLET, NEUMANN = 1, 2

BASE = {"op": "", "D": 3, "n": 16, "p": 2, "nu": 1e-6, "noise": 0.0, "prec": 0, "block": False, "falgout": 0, "distance": 1,
        "relax": "FCF", "theta": 0.25, "theta_r": -1.0, "rtol": 1e-8, "k": 1, "dtype": "float64"}


def _case(name, op, **kw):
    return dict(BASE, name=name, op=op, **kw)


def listed():
    return [
        # the preconditioner of a small 1D + time problem, inside a user's own Krylov loop: launches and latency
        _case("vcycle_small", "vcycle", D=2, n=32, p=1, nu=1e-4),
        # the same for an ordinary 2D + time problem, in the benchmarked form (FP32 hierarchy, facet blocks)
        _case("vcycle_mid", "vcycle", n=16, prec=1, block=True),
        # the benchmark's mesh and degree: 7.9 million unknowns, far larger than the L2
        _case("vcycle_large", "vcycle", n=48, prec=1, block=True, falgout=8192),
        # one hierarchy, many right-hand sides (uncertainty ensembles, several sources)
        _case("vcycle_many", "vcycle_multi", n=20, prec=1, k=32, dtype="float32"),
        # the whole call on a small system with the default options: one time-to-solution of a 1D + time study
        _case("solve_small", "solve", D=2, n=32, p=1, nu=1e-4),
        # the headline step (sequential first pass, FP32 hierarchy, FP64 FGMRES) on an ordinary mesh
        _case("solve_mid", "solve", n=16, prec=1, block=True),
        # the same step with the blocked splitting on a mesh eight times as large
        _case("solve_blocked", "solve", n=32, prec=1, block=True, falgout=8192),
        # another right-hand side on a hierarchy that is kept, on a large mesh: FGMRES(30) alone
        _case("gmres_large", "gmres", n=40, prec=1, block=True, falgout=8192),
        # the paper's own solver: BiCGSTAB to 1e-12, strength pair, forward Gauss-Seidel on F, then on all points
        _case("paper_solver", "bicgstab", n=15, p=1, theta=0.2, theta_r=0.3, falgout=1024, relax="fa", rtol=1e-12),
        # assembly of the trace system, quadratic elements
        _case("assemble_p2", "assemble", n=24),
        # assembly with cubic elements on an odd mesh
        _case("assemble_p3", "assemble", n=17, p=3, nu=1e-5),
        # the backward half of one optimisation step: adjoint setup and solve, velocity gradient
        _case("adjoint_step", "adjoint", n=20, nu=1e-4, noise=0.1, prec=1, block=True, falgout=8192),
    ]


def draw(rng):
    """One more case of the same ranges; the largest sizes of each call are those of the listed cases."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["vcycle", "vcycle", "vcycle_multi", "solve", "solve", "gmres", "bicgstab", "assemble", "adjoint"])
    D = 2 if rng.random() < 0.3 and op in ("vcycle", "solve", "gmres", "assemble") else 3
    p = rng.choice([1, 2, 3])
    nu = 10.0 ** rng.uniform(-6.0, -4.0)
    kw = dict(D=D, p=p, nu=nu, prec=rng.choice([0, 1, 1, 2]), block=rng.random() < 0.7, falgout=rng.choice([0, 1024, 8192]))
    top = {1: 1.25, 2: 1.0, 3: 0.75}[p]          # about the same unknowns at every degree
    if D == 2:
        return _drop(op, **dict(kw, n=size(9, 150 * top)))
    if op == "vcycle":
        return _drop(op, **dict(kw, n=size(5, 36 * top), falgout=8192 if rng.random() < 0.5 else 1024))
    if op == "vcycle_multi":
        dtype = rng.choice(["float32", "float64"])
        return _drop(op, **dict(kw, n=size(5, 18 * top), prec=int(dtype == "float32"), k=rng.randint(2, 32), dtype=dtype))
    if op == "solve":
        if rng.random() < 0.25:                  # the diffusive end needs distance-two neighbourhoods
            return _drop(op, **dict(kw, n=size(4, 10), p=min(p, 2), nu=1e-2, distance=2, falgout=0, prec=0))
        return _drop(op, **dict(kw, n=size(5, 14 * top) if kw["falgout"] == 0 else size(5, 30 * top)))
    if op == "gmres":
        return _drop(op, **dict(kw, n=size(8, 34 * top), falgout=8192))
    if op == "bicgstab":
        return _drop(op, **dict(kw, n=size(4, 12 * top), theta=0.2, theta_r=0.3, relax=rng.choice(["fa", "FCF"]),
                                falgout=1024, prec=0, rtol=1e-12))
    if op == "assemble":
        return _drop(op, **dict(kw, n=size(4, 24 if p < 3 else 17)))
    return _drop(op, **dict(kw, n=size(4, 18 * top), nu=1e-4, noise=0.1, prec=rng.choice([0, 1]), falgout=8192))


def _drop(op, **kw):
    c = dict(BASE, op=op, **kw)
    if op == "assemble":                         # nothing of a hierarchy is in it
        c.update(prec=0, block=False, falgout=0)
    return c


# ---------------------------------------------------------------- inputs
def _reflect(D):
    return choose_reflection(D, [1.0] if D == 2 else [0.0, 0.0])


@functools.lru_cache(maxsize=16)
def _mesh(D, n):
    return hdg.HdgMesh.from_mesh(build_mesh(D, n, reflect=_reflect(D)), DEV)


@functools.lru_cache(maxsize=8)
def _tables(D, p):
    return hdg.HdgTables(D, p, DEV)


def _problem(c, seed):
    """Mesh, tables and problem data at the quadrature points.  2D + time: a rotation about a point near the middle
    (plus a normal deviation per element when noise is set); 1D + time: a velocity near one.  The data are those of
    a smooth travelling field whose phases come from the seed."""
    D, n, p = c["D"], c["n"], c["p"]
    mesh, tab = _mesh(D, n), _tables(D, p)
    r = np.random.default_rng([seed, D, n, p])
    w, s1, s2 = r.uniform(0.9, 1.1), r.uniform(0.0, 0.3), r.uniform(0.0, 0.3)
    cx, cy = 0.5 + r.uniform(-0.03, 0.03, 2)
    xv, xf, xF = hdg.points(mesh, tab)

    if D == 3:
        def vel(X):
            return torch.stack([-w * (X[..., 2] - cy), w * (X[..., 1] - cx)], -1)

        def u(X):
            return torch.sin(PI * X[..., 1] + s1) * torch.sin(PI * X[..., 2] + s2) * torch.cos(2 * PI * X[..., 0])

        def src(X):
            t, sx, sy = 2 * PI * X[..., 0], torch.sin(PI * X[..., 1] + s1), torch.sin(PI * X[..., 2] + s2)
            gx = PI * torch.cos(PI * X[..., 1] + s1) * sy * torch.cos(t)
            gy = PI * sx * torch.cos(PI * X[..., 2] + s2) * torch.cos(t)
            a = vel(X)
            return -2 * PI * sx * sy * torch.sin(t) + a[..., 0] * gx + a[..., 1] * gy + c["nu"] * 2 * PI * PI * u(X)
    else:
        def vel(X):
            return torch.full(X.shape[:-1] + (1,), w, dtype=X.dtype, device=X.device)

        def u(X):
            return torch.sin(2 * PI * X[..., 1] + s1) * torch.exp(-X[..., 0])

        def src(X):
            e = torch.exp(-X[..., 0])
            s, k = torch.sin(2 * PI * X[..., 1] + s1), torch.cos(2 * PI * X[..., 1] + s1)
            return e * (-s + w * 2 * PI * k + c["nu"] * 4 * PI * PI * s)

    vv, vf = vel(xv), vel(xf)
    if c["noise"] > 0.0:
        g = torch.Generator(device=DEV).manual_seed(seed)
        dev = c["noise"] * torch.randn((mesh.n_elems, D - 1), generator=g, device=DEV, dtype=torch.float64)
        vv, vf = vv + dev[:, None, :], vf + dev[:, None, None, :]
    data = hdg.HdgData(c["nu"], 10.0 * p * p, vv.contiguous(), vf.contiguous(), src(xv).contiguous(), u(xf).contiguous(),
                       u(xF).contiguous())
    return mesh, tab, data


def _options(c, tab):
    return dict(theta=c["theta"], theta_r=c["theta_r"], distance=c["distance"], precision=c["prec"],
                falgout_block=c["falgout"], relax=c["relax"], block_size=tab.b if c["block"] else 0)


def prepare(case, seed):
    c = dict(BASE, **case)
    mesh, tab, data = _problem(c, seed)
    s = {"c": c, "mesh": mesh, "tab": tab, "data": data, "opts": _options(c, tab)}
    if c["op"] == "assemble":
        return s
    s["sys"] = sy = hdg.assemble(mesh, tab, data)
    s["A"], s["b"] = sy.A, sy.rhs
    g = torch.Generator(device=DEV).manual_seed(seed + 1)
    if c["op"] != "adjoint":
        del s["data"]                            # the assembly's inputs are not kept by a program that only solves
    if c["op"] == "adjoint":
        H = air.setup(sy.A, **s["opts"])
        s["u"], _ = air.gmres_solve(sy.A, H, sy.rhs, rtol=c["rtol"])
        noise = torch.randn(sy.A.n, generator=g, device=DEV, dtype=torch.float64)
        s["g"] = 0.1 * s["u"] + 0.01 * noise     # dL/du of a misfit
        H.free()
    elif c["op"] in ("gmres", "bicgstab"):
        s["H"] = air.setup(sy.A, **s["opts"])
    elif c["op"] == "vcycle":
        s["H"] = air.setup(sy.A, **s["opts"])
        s["b"] = torch.randn(sy.A.n, generator=g, device=DEV, dtype=torch.float64)
    elif c["op"] == "vcycle_multi":
        s["H"] = air.setup(sy.A, **s["opts"])
        s["b"] = torch.randn((sy.A.n, c["k"]), generator=g, device=DEV, dtype=getattr(torch, c["dtype"]))
    return s


# ---------------------------------------------------------------- one pass
def run(state):
    s, c = state, state["c"]
    op = c["op"]
    if op == "vcycle":
        return s["H"].vcycle(s["b"])
    if op == "vcycle_multi":
        return air.vcycle_multi(s["H"], s["b"])
    if op == "solve":
        H = air.setup(s["A"], **s["opts"])
        x, _ = air.gmres_solve(s["A"], H, s["b"], rtol=c["rtol"])
        return x
    if op == "gmres":
        x, _ = air.gmres_solve(s["A"], s["H"], s["b"], rtol=c["rtol"])
        return x
    if op == "bicgstab":
        x, _ = air.bicgstab_solve(s["A"], s["H"], s["b"], rtol=c["rtol"])
        return x
    if op == "assemble":
        y = hdg.assemble(s["mesh"], s["tab"], s["data"])
        return {"row_ptr": y.A.row_ptr, "col": y.A.col, "val": y.A.val, "rhs": y.rhs, "diag": y.diag, "lam_dir": y.lam_dir}
    sy, b = s["sys"], s["tab"].b
    At = air.transpose_scaled(sy.A, b, sy.diag)
    Ht = air.setup(At, **s["opts"])
    y, _ = air.gmres_solve(At, Ht, air.block_diag_apply(b, sy.diag, 3, s["g"]), rtol=c["rtol"])
    lam = air.block_diag_apply(b, sy.diag, 1, y)
    grad = hdg.velocity_gradient(s["mesh"], s["tab"], s["data"], sy, s["u"], lam)
    return {"adjoint": lam, "gradient": grad}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Finest level only (the coarse levels follow from it).  A row of the scaled operator holds one diagonal entry and
    2 D whole facet blocks; stored, an entry is its value and its share of a block's column index."""
    c = dict(BASE, **case)
    D, n, p = c["D"], c["n"], c["p"]
    b = math.comb(p + D - 1, D - 1)
    nb = math.comb(p + D, D)
    elems = math.factorial(D) * n ** D
    free = 12 * n ** 3 - 2 * n * n if D == 3 else 3 * n * n
    rows = free * b
    nnz = rows * (1 + 2 * D * b)
    wide = {0: 8, 1: 4, 2: 2}[c["prec"]]
    stored = nnz * (wide + 4.0 / b)
    csr = 12 * nnz + 8 * rows
    if c["op"] == "vcycle":
        return {"bytes": stored + 16 * rows, "flops": 4 * nnz}
    if c["op"] == "vcycle_multi":
        w = 4 if c["dtype"] == "float32" else 8
        return {"bytes": nnz * (w + 4.0 / b) + 2 * w * c["k"] * rows, "flops": 4 * nnz * c["k"]}
    if c["op"] in ("solve", "gmres", "bicgstab"):
        return {"bytes": csr + 16 * rows, "flops": 4 * nnz}
    nq, nqf, nt = (p + 2) ** D, (p + 2) ** (D - 1), (D + 1) * b
    inputs = 8 * elems * (nq * D + (D + 1) * nqf * D)
    local = elems * (2 * nq * nb * (nb + D) + 2 * (D + 1) * nqf * (nb * nb + 2 * nb * b + b * b) + 2 * nb * nb * (nb / 3 + nt)
                     + 2 * nt * nt * nb)
    if c["op"] == "assemble":
        return {"bytes": inputs + csr + 8 * rows * (1 + b), "flops": local}
    return {"bytes": inputs + 2 * csr + 32 * rows, "flops": 2 * local + 4 * nnz}


# ---------------------------------------------------------------- the same in 64 bits, by torch
def _sparse(rp, ci, v, shape):
    t = [torch.as_tensor(x).to(DEV) for x in (rp, ci, v)]
    return torch.sparse_csr_tensor(t[0].long(), t[1].long(), t[2].double(), size=shape)


def _levels(H):
    """The hierarchy's operators: what the V-cycle applies."""
    out, last = [], H.levels() - 1
    for l in range(last + 1):
        i = H.info(l)
        L = {"A": _sparse(H.export(l, "A.row_ptr"), H.export(l, "A.col"), H.export(l, "A.val"), (i.n, i.n))}
        if l < last:
            L["R"] = _sparse(H.export(l, "R.row_ptr"), H.export(l, "R.col"), H.export(l, "R.val"), (i.nc, i.n))
            cf, pc = (torch.as_tensor(H.export(l, w)).to(DEV) for w in ("cf", "pcol"))
            L["C"], L["pcol"] = cf == 1, pc.long()
            r, k, v = torch.as_tensor(H.export(l, "A.row_ptr")).to(DEV), L["A"].col_indices(), L["A"].values()
            rows = torch.repeat_interleave(torch.arange(i.n, device=DEV), r[1:] - r[:-1])
            d = torch.zeros(i.n, dtype=torch.float64, device=DEV)
            d[rows[rows == k]] = v[rows == k]
            L["d"] = d[:, None]
        else:
            L["lu"] = torch.linalg.lu_factor(L["A"].to_dense())
        out.append(L)
    return out


def _vcycle64(levels, b, relax="FCF"):
    """x = V(b), columns of b at once: a zero guess, restriction, coarsest solve, interpolation, Jacobi sweeps."""
    bs = [b]
    for L in levels[:-1]:
        bs.append(L["R"] @ bs[-1])
    x = torch.linalg.lu_solve(*levels[-1]["lu"], bs[-1])
    for L, r in zip(reversed(levels[:-1]), reversed(bs[:-1])):
        pc = L["pcol"]
        x = torch.where((pc >= 0)[:, None], x[pc.clamp(min=0)], torch.zeros((), dtype=torch.float64, device=DEV))
        for ch in relax:
            on = L["C"] if ch == "C" else ~L["C"]
            x = torch.where(on[:, None], x + (r - L["A"] @ x) / L["d"], x)
    return x


def _solve64(A, b, levels, tol=2e-14, cycles=20, m=40):
    """A x = b by restarted flexible GMRES in 64 bits until the true residual is at rounding level.  The levels only
    speed it up: the answer does not depend on them."""
    x, bn, best = torch.zeros_like(b), b.norm(), None
    for _ in range(cycles):
        r = b - (A @ x[:, None])[:, 0]
        rel = float(r.norm() / bn)
        if best is not None and rel > 0.5 * best[0] and best[0] < 1e-12:
            break
        if best is None or rel < best[0]:
            best = (rel, x.clone())
        if rel <= tol:
            break
        beta = r.norm()
        V, Z, Hm = [r / beta], [], np.zeros((m + 1, m))
        k = 0
        for j in range(m):
            Z.append(_vcycle64(levels, V[j][:, None])[:, 0])
            w = (A @ Z[j][:, None])[:, 0]
            for _twice in range(2):
                for i in range(j + 1):
                    h = float(V[i] @ w)
                    Hm[i, j] += h
                    w = w - h * V[i]
            Hm[j + 1, j] = float(w.norm())
            k = j + 1
            e = np.zeros(k + 1)
            e[0] = float(beta)
            y, res, _, _ = np.linalg.lstsq(Hm[:k + 1, :k], e, rcond=None)
            if Hm[j + 1, j] <= 1e-300 or np.linalg.norm(e - Hm[:k + 1, :k] @ y) <= 1e-8 * float(beta):
                break
            V.append(w / Hm[j + 1, j])
        for i in range(k):
            x = x + float(y[i]) * Z[i]
    return best[1]


def _elements64(mesh, tab, data, lo, hi, dvel=None):
    """Condensed element matrices S_K (E, nt, nt) and H_K (E, nt) of elements lo..hi; dvel is added to the velocity."""
    r, D = tab.ref, mesh.D
    T = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64)).to(DEV)  # noqa: E731
    el = mesh.elems[lo:hi].long()
    X = mesh.verts[el]
    E, nb, b = hi - lo, r.nb, r.b
    J = (X[:, 1:] - X[:, :1]).transpose(1, 2)
    Ji, det = torch.linalg.inv(J), torch.linalg.det(J).abs()
    h = torch.stack([(X[:, i] - X[:, j]).norm(dim=-1) for i in range(D + 1) for j in range(i)]).amax(0)
    nu, pen = data.nu, data.nu * data.alpha / h
    phi, gphi, psi, wq, wf = T(r.phi), T(r.gphi), T(r.psi), T(r.wq), T(r.wf)
    a = data.vel_vol[lo:hi]
    af = data.vel_face[lo:hi]
    if dvel is not None:
        a, af = a + dvel[:, None, :], af + dvel[:, None, None, :]
    W = det[:, None] * wq
    ah = torch.cat([torch.ones_like(a[..., :1]), a], -1)
    adv = torch.einsum("eqk,qik->eqi", torch.einsum("ekd,eqd->eqk", Ji, ah), gphi)
    A = -torch.einsum("eqi,eqj->eij", adv, W[..., None] * phi)
    gs = torch.einsum("eks,qik->eqis", Ji[:, :, 1:], gphi).reshape(E, len(wq), nb, D - 1)
    A = A + nu * torch.einsum("eqis,eqjs->eij", gs * W[..., None, None], gs)
    Fv = (W * data.src[lo:hi]) @ phi
    B, C, Dm, Gv = [], [], torch.zeros((E, (D + 1) * b, (D + 1) * b), dtype=torch.float64, device=DEV), []
    lookup = {tuple(q): i for i, q in enumerate(r.perms.tolist())}
    code = torch.zeros(D ** D, dtype=torch.long, device=DEV)
    for q, i in lookup.items():
        code[sum(v * D ** m for m, v in enumerate(q))] = i
    gb = torch.cat([-torch.ones((1, D), dtype=torch.float64), torch.eye(D, dtype=torch.float64)]).to(DEV)
    for k in range(D + 1):
        loc = [j for j in range(D + 1) if j != k]
        order = torch.argsort(el[:, loc], dim=1)
        pi = code[(order * torch.tensor([D ** m for m in range(D)], device=DEV)).sum(1)]
        ph, gp = T(r.phi_f[k])[pi], T(r.gphi_f[k])[pi]
        gl = torch.einsum("ekd,k->ed", Ji, gb[k])
        gn = gl.norm(dim=-1)
        nrm = -gl / gn[:, None]
        Wf = (det * gn)[:, None] * wf              # area (D-1)! = D (det / D!) |grad| (D-1)!
        an = nrm[:, :1] + torch.einsum("eqd,ed->eq", af[:, k], nrm[:, 1:])
        up, dn = 0.5 * (an + an.abs()), 0.5 * (an - an.abs())
        ns = torch.cat([torch.zeros_like(nrm[:, :1]), nrm[:, 1:]], -1)
        dnorm = torch.einsum("eqik,ek->eqi", gp, torch.einsum("ekd,ed->ek", Ji, ns))
        pw = Wf[..., None] * ph
        A = A + torch.einsum("eqi,eqj->eij", pw * (up + pen[:, None])[..., None], ph)
        t = torch.einsum("eqi,eqj->eij", pw, dnorm)
        A = A - nu * (t + t.transpose(1, 2))
        dw = nu * Wf[..., None] * dnorm
        B.append(torch.einsum("eqi,qm->eim", pw * (dn - pen[:, None])[..., None] + dw, psi))
        C.append(torch.einsum("eqj,qm->emj", dw - pw * (up + pen[:, None])[..., None], psi))
        neu = (mesh.facet_kind[mesh.elem_facets[lo:hi, k].long()] == NEUMANN).double()[:, None]
        Dm[:, k * b:(k + 1) * b, k * b:(k + 1) * b] = torch.einsum("eql,qm->eml", (Wf * (neu * up - dn + pen[:, None]))[..., None] * psi, psi)
        gN = torch.where(an < 0.0, -an * data.u0_face[lo:hi, k], torch.zeros_like(an)) * neu
        Gv.append((Wf * gN) @ psi)
    B, C, Gv = torch.cat(B, 2), torch.cat(C, 1), torch.cat(Gv, 1)
    Y = torch.linalg.solve(A, torch.cat([B, Fv[:, :, None]], 2))
    return Dm - C @ Y[:, :, :-1], Gv - (C @ Y[:, :, -1:])[..., 0]


def _assemble64(mesh, tab, data):
    """The scaled system's values in the layout of the assembled one, and what comes with it."""
    D, b, F = mesh.D, tab.b, mesh.n_facets
    free = mesh.facet_kind != DIRICHLET
    Ff = int(free.sum())
    num = torch.cumsum(free, 0) - 1
    f = D + 1
    dp, W = torch.as_tensor(tab.ref.dir_proj).to(DEV), ~free
    lam = torch.zeros((F, b), dtype=torch.float64, device=DEV)
    lam[W] = data.g_dir[W] @ dp.T
    Sd = torch.zeros((F, b, b), dtype=torch.float64, device=DEV)
    Hf = torch.zeros((F, b), dtype=torch.float64, device=DEV)
    fa, ga, bl = [], [], []
    for lo in range(0, mesh.n_elems, 16384):
        hi = min(mesh.n_elems, lo + 16384)
        S, Hk = _elements64(mesh, tab, data, lo, hi)
        S = S.reshape(hi - lo, f, b, f, b).transpose(2, 3)
        ef = mesh.elem_facets[lo:hi].long()
        for k in range(f):
            Hf.index_add_(0, ef[:, k], Hk[:, k * b:(k + 1) * b])
            Sd.index_add_(0, ef[:, k], S[:, k, k])
            for q in range(f):
                if q != k:
                    on = free[ef[:, k]] & ~free[ef[:, q]]
                    Hf.index_add_(0, ef[on, k], -(S[on, k, q] @ lam[ef[on, q]][..., None])[..., 0])
                    on = free[ef[:, k]] & free[ef[:, q]]
                    fa.append(num[ef[on, k]])
                    ga.append(num[ef[on, q]])
                    bl.append(S[on, k, q])
    fa, ga, bl = torch.cat(fa), torch.cat(ga), torch.cat(bl)
    Sd, Hf = Sd[free], Hf[free]
    rhs = torch.linalg.solve(Sd, Hf[..., None]).reshape(-1)
    bl = torch.linalg.solve(Sd[fa], bl)
    order = torch.argsort(fa * Ff + ga)
    fa, ga, bl = fa[order], ga[order], bl[order]
    cnt = torch.bincount(fa, minlength=Ff)
    before = torch.bincount(fa[ga < fa], minlength=Ff)
    start = torch.cumsum(cnt, 0) - cnt
    rowlen = cnt * b + 1
    base = torch.cumsum(rowlen * b, 0) - rowlen * b        # first entry of a facet's rows
    ii = torch.arange(b, device=DEV)
    rank = torch.arange(len(fa), device=DEV) - start[fa]
    pos = (base[fa] + rank * b + (ga > fa))[:, None, None] + rowlen[fa][:, None, None] * ii[None, :, None] + ii
    val = torch.empty(int((rowlen * b).sum()), dtype=torch.float64, device=DEV)
    val[pos.reshape(-1)] = bl.reshape(-1)
    val[((base + before * b)[:, None] + rowlen[:, None] * ii).reshape(-1)] = 1.0
    return {"row_ptr": None, "col": None, "val": val, "rhs": rhs, "diag": Sd, "lam_dir": lam}


def _transposed64(A):
    rows = torch.repeat_interleave(torch.arange(A.n, device=DEV), A.row_ptr[1:] - A.row_ptr[:-1])
    t = torch.sparse_coo_tensor(torch.stack([A.col.long(), rows]), A.val, (A.n, A.n)).coalesce()
    return t.to_sparse_csr()


def exact(case, seed):
    """V-cycle: the exported operators applied in 64 bits.  Solves: the solution itself.  Assembly and gradient: the
    bilinear form, and its derivative by autograd."""
    s = prepare(case, seed)
    c = s["c"]
    op = c["op"]
    if op == "vcycle":
        return _vcycle64(_levels(s["H"]), s["b"][:, None], c["relax"])[:, 0]
    if op == "vcycle_multi":
        return _vcycle64(_levels(s["H"]), s["b"].double(), c["relax"])
    if op == "assemble":
        return _assemble64(s["mesh"], s["tab"], s["data"])
    helper = dict(s["opts"], relax="FCF", precision=0)
    if op in ("solve", "gmres", "bicgstab"):
        lv = _levels(air.setup(s["A"], **helper))
        return _solve64(lv[0]["A"], s["b"], lv)
    sy, b = s["sys"], s["tab"].b
    At = _transposed64(sy.A)
    Ht = air.setup(air.CSR(At.crow_indices(), At.col_indices().int(), At.values(), sy.A.n), **helper)
    lam = _solve64(At, s["g"], _levels(Ht))
    mesh, tab, data = s["mesh"], s["tab"], s["data"]
    free = mesh.facet_kind != DIRICHLET
    full = sy.lam_dir.clone()
    full[free] = s["u"].reshape(-1, b)
    mu = torch.zeros_like(full)
    mu[free] = torch.linalg.solve(sy.diag.transpose(1, 2), lam.reshape(-1, b, 1))[..., 0]
    grads = []
    for lo in range(0, mesh.n_elems, 8192):
        hi = min(mesh.n_elems, lo + 8192)
        dv = torch.zeros((hi - lo, mesh.D - 1), dtype=torch.float64, device=DEV, requires_grad=True)
        S, Hk = _elements64(mesh, tab, data, lo, hi, dv)
        ef = mesh.elem_facets[lo:hi].long()
        lk, mk = full[ef].reshape(hi - lo, -1), mu[ef].reshape(hi - lo, -1)
        ((mk * Hk).sum() - (mk * (S @ lk[..., None])[..., 0]).sum()).backward()
        grads.append(dv.grad)
    return {"adjoint": lam, "gradient": torch.cat(grads)}

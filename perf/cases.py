"""The workloads this library is measured on, through its public entry points: whole solves on
the plane and the cubed sphere (FP64 and with the FP32 preconditioner, degree 0 to 3), a batch of
uneven solves, the set-up after new coefficients, the S apply and the line smoother on their own,
and one training gradient of the learned coarse map. `exact` restates the discretisation in plain
torch FP64 (nothing of the library runs in it; only its input meshes are shared)."""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2210_11797_gb300 import hmg
from paper_2210_11797_gb300 import inputs as I

_SPHERE = dict(mesh="sphere", precision="fp64", degree=0, tol=1e-6, background="isothermal", omega=0.0, tuned=False)
_PLANE = dict(mesh="plane", precision="fp64", degree=0, tol=1e-10, background="unit", omega=0.0, tuned=False)


def listed():
    return [
        # the smallest solve in use: the planar Helmholtz test problem (latency of one solve call)
        dict(_PLANE, name="solve_plane16", kind="solve", n=16, nlev=8),
        # a development-size sphere with a rotating, stratified background: solve and recovery
        dict(_SPHERE, name="solve_c24_rotating", kind="solve", n=24, nlev=30, background="stratified",
             omega=I.EARTH_OMEGA),
        # the paper's mesh, one implicit solve of a time step, FP64, tuned once as a long run does
        dict(_SPHERE, name="solve_c96", kind="solve", n=96, nlev=30, tuned=True),
        # the same time step with the FP32 preconditioner
        dict(_SPHERE, name="solve_c96_mixed", kind="solve", n=96, nlev=30, precision="mixed", tuned=True),
        # an ensemble: uneven members solved together in one call
        dict(name="batch12_mixed", kind="batch", count=12, first=0, nmax=48, precision="mixed", tol=1e-6),
        # a new time step's background: the operators rebuilt, then the first right-hand side
        dict(_SPHERE, name="setup_c96", kind="setup", n=96, nlev=30, background="stratified", omega=I.EARTH_OMEGA),
        # operator application alone (a user's own Krylov method), levels not a multiple of a warp
        dict(_SPHERE, name="apply_c64x37", kind="apply", n=64, nlev=37),
        # the line smoother alone (Algorithm 1 as a preconditioner), tall columns
        dict(_SPHERE, name="smooth_c48x50", kind="smooth", n=48, nlev=50, sweeps=3),
        # higher order: the degree-1 system solved in FP64
        dict(_PLANE, name="solve_degree1", kind="solve", n=64, nlev=16, degree=1, tol=1e-6),
        # the degree-3 system with the FP32 preconditioner
        dict(_PLANE, name="solve_degree3_mixed", kind="solve", n=16, nlev=16, degree=3, precision="mixed"),
        # set-up of the degree-3 system (304 x 304 cell matrices), right-hand side and recovery
        dict(_PLANE, name="setup_degree3", kind="setup", n=12, nlev=8, degree=3),
        # one minibatch of the learned coarse map's training: forward and backward
        dict(name="grad_64x16x16", kind="grad", nsamp=64, nx=16, ny=16, nlev=30),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve_p", "setup", "setup_p", "apply", "smooth", "batch", "grad"])
    precision = rng.choice(["fp64", "mixed"])
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(3, 12), first=rng.randint(0, 52), nmax=48, precision=precision,
                    tol=1e-6)
    if kind == "grad":
        return dict(kind="grad", nsamp=_log(rng, 1, 64), nx=rng.randint(4, 16), ny=rng.randint(4, 16),
                    nlev=rng.randint(8, 30))
    if kind in ("solve_p", "setup_p"):
        p = rng.randint(1, 3)
        n = 4 * _log(rng, 1, {1: 16, 2: 8, 3: 4}[p]) if kind == "solve_p" else _log(rng, 2, {1: 48, 2: 24, 3: 12}[p])
        return dict(_PLANE, kind=kind[:5], n=n, nlev=rng.randint(2, 16 if kind == "solve_p" else 8), degree=p,
                    precision=precision if kind == "solve_p" else "fp64")
    if rng.random() < 0.3:
        return dict(_PLANE, kind=kind, n=4 * _log(rng, 2, 32), nlev=rng.randint(3, 40),
                    precision=precision if kind == "solve" else "fp64", **({"sweeps": rng.randint(1, 4)} if kind == "smooth" else {}))
    n, bg = 4 * _log(rng, 2, 20), rng.choice(["isothermal", "stratified"])
    c = dict(_SPHERE, kind=kind, n=n, nlev=_log(rng, 5, 70 if n <= 56 else 36), background=bg,
             omega=rng.choice([0.0, I.EARTH_OMEGA]))
    if kind == "solve":
        c.update(precision=precision, tuned=rng.random() < 0.3)
    if kind == "smooth":
        c["sweeps"] = rng.randint(1, 4)
    return c


# ---- inputs -----------------------------------------------------------------------------------
@functools.lru_cache(maxsize=64)
def _hierarchy(mesh, n, nlev):
    levels = I.mg_levels_for(n, 2 if mesh == "plane" and n <= 16 else 4)
    if mesh == "plane":
        return I.planar_hierarchy(n, nlev, 1.0, I.uniform_levels(nlev, 0.1), levels)
    return I.sphere_hierarchy(n, nlev, I.quadratic_levels(nlev, 30000.0), levels)


@functools.lru_cache(maxsize=64)
def _system(mesh, n, nlev, background, omega):
    hier = _hierarchy(mesh, n, nlev)
    if background == "unit":
        co = I.Coefficients([I.unit_background(m) for m in hier.meshes], preset=1, sigma=1.0 / 0.05 ** 2)
    else:
        make = I.stratified_background if background == "stratified" else I.isothermal_background
        co = I.Coefficients([make(m) for m in hier.meshes], dt=I.acoustic_dt(n, 8.0), omega=omega)
    return hier, co


def _of(case):
    return _system(case["mesh"], case["n"], case["nlev"], case["background"], case["omega"])


def _members(case):
    sizes = [s for s in I.batched_sizes(64, 3)[case["first"]:case["first"] + case["count"]] if s[0] <= case["nmax"]]
    return [dict(_SPHERE, n=n, nlev=L) for n, L in sizes]


def _sizes(case):
    """Cells, trace unknowns, velocity and pressure dofs per cell."""
    ncol = (6 if case["mesh"] == "sphere" else 1) * case["n"] ** 2
    L, p = case["nlev"], case["degree"]
    return ncol * L, (p + 1) ** 2 * ncol * (3 * L + 1), 3 * (p + 1) ** 2 * (p + 2), (p + 1) ** 3


def _normals(seed, *shapes, dtype=torch.float64):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    return [torch.randn(s, generator=g, dtype=dtype, device=dev) for s in shapes]


def _data(case, seed):
    """R_u, R_Pi, two trace vectors and a cell vector."""
    C, T, nu, npr = _sizes(case)
    return _normals(seed, C * nu, C * npr, T, T, C)


def _patches(case, seed):
    x, t = _normals(seed, (case["nsamp"], case["nx"] * case["ny"], case["nlev"]),
                    (case["nsamp"], case["nx"] * case["ny"], case["nlev"]), dtype=torch.float32)
    return x, t, I.flatten_coarse_model(I.coarse_model_init(seed % 1000))


def _solver(case):
    hier, co = _of(case)
    return hmg.Solver(hier, co, tol=case["tol"], precision=case["precision"], degree=case["degree"])


def prepare(case, seed):
    st = dict(case=case)
    if case["kind"] == "batch":
        ms = _members(case)
        st["solvers"] = [_solver(dict(m, precision=case["precision"], tol=case["tol"])) for m in ms]
        data = [_data(m, seed + 1000 * i) for i, m in enumerate(ms)]
        st["Ru"], st["Rp"], st["lam"] = [d[0] for d in data], [d[1] for d in data], [torch.empty_like(d[2]) for d in data]
        return st
    if case["kind"] == "grad":
        plane = dict(_PLANE, n=4, nlev=case["nlev"])
        st["solver"] = _solver(plane)
        st["x"], st["t"], w = _patches(case, seed)
        st["solver"].set_coarse_model(w)
        return st
    st["solver"] = _solver(case)
    st["Ru"], st["Rp"], st["x"], st["b"], st["c"] = _data(case, seed)
    if case["tuned"]:
        st["solver"].autotune()
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "batch":
        return hmg.solve_batched(st["solvers"], st["Ru"], st["Rp"], st["lam"])[0]
    s = st["solver"]
    if kind == "solve":
        lam, _stats = s.solve(st["Ru"], st["Rp"])
        u, pi = s.reconstruct(lam, st["Ru"], st["Rp"])
        return {"lam": lam, "u": u, "pi": pi}
    if kind == "setup":
        s.assemble()
        out = {"B": s.trace_rhs(st["Ru"], st["Rp"]), "Sx": s.apply_trace(st["x"]), "gamma": s.gamma()}
        if case["degree"] == 0:
            out["Hc"] = s.apply_pressure(0, st["c"])
        else:
            out["u"], out["pi"] = s.reconstruct(st["x"], st["Ru"], st["Rp"])
        return out
    if kind == "apply":
        return s.apply_trace(st["x"])
    if kind == "smooth":
        return s.line_smooth(st["b"], st["x"].clone(), case["sweeps"])
    loss, g = s.coarse_model_grad(st["x"], st["t"], case["nx"], case["ny"])
    return {"loss": loss, "grad": g}


# ---- what a pass cannot do without --------------------------------------------------------------
def _solve_work(case):
    """Reading the cell residuals and the inverse cell matrices, writing lambda, u and Pi; then per
    iteration (as many as the workload takes) two applies of S and two preconditioner calls: three
    passes over S (two sweeps, one residual), the pressure multigrid's coefficients and the vectors."""
    C, T, nu, npr = _sizes(case)
    nb = (case["degree"] + 1) ** 2
    w = 4 if case["precision"] == "mixed" else 8
    per_row = 11 * nb
    its = {"sphere": 6, "plane": 9}[case["mesh"]] if case["degree"] == 0 else 12 + 4 * case["degree"]
    once = 8 * (C * (nu + npr) ** 2 + 3 * C * (nu + npr) + 3 * T)
    apply = 8 * T * (per_row + 2)
    precond = 3 * w * T * (per_row + 3) + 40 * w * C
    return {"bytes": once + its * 2 * (apply + precond),
            "flops": 2 * C * (nu + npr) ** 2 + its * 2 * (2 * T * per_row * 4 + 60 * C)}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        ws = [_solve_work(dict(m, precision=case["precision"])) for m in _members(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    if kind == "solve":
        return _solve_work(case)
    if kind == "grad":
        cells = case["nsamp"] * case["nx"] * case["ny"] * case["nlev"]
        return {"bytes": 8 * cells, "flops": 3 * 2 * 3360 * cells}
    C, T, nu, npr = _sizes(case)
    N, nb = nu + npr, (case["degree"] + 1) ** 2
    S = 8 * 11 * nb * T
    if kind == "setup":   # the inverse cell matrices and the rows of S written, then read once
        return {"bytes": 2 * (8 * C * N * N + S) + 8 * (4 * C * N + 3 * T), "flops": 2 * C * N ** 3 + 4 * C * N * N}
    if kind == "apply":
        return {"bytes": S + 16 * T, "flops": 22 * T}
    return {"bytes": case["sweeps"] * (S + 32 * T), "flops": case["sweeps"] * 30 * T}


# ---- the same in plain FP64 ----------------------------------------------------------------------
def _t(a, like):
    return torch.as_tensor(np.ascontiguousarray(a), device=like.device)


class _Cells:
    """Degree 0: per-cell inverse blocks and the trace numbering of the finest mesh."""

    def __init__(self, case, like):
        hier, co = _of(case)
        m, bg = hier.meshes[0], co.levels[0]
        self.L, self.ncol, L = m.nlev, m.ncol, m.nlev
        f8 = lambda a: _t(np.asarray(a, np.float64), like)
        i8 = lambda a: _t(np.asarray(a, np.int64), like)
        z, ce = f8(m.z_levels), i8(m.col_edges)
        col = torch.arange(m.ncol, device=like.device).repeat_interleave(L)
        lev = torch.arange(L, device=like.device).repeat(m.ncol)
        self.col, self.lev = col, lev
        NH = m.nedge * L
        zb = NH + col * (L + 1) + lev
        self.g = torch.stack([ce[col, f] * L + lev for f in range(4)] + [zb, zb + 1], 1)
        self.T, self.NH = NH + m.ncol * (L + 1), NH
        corners = f8(m.corners)[:, [0, 1, 3, 2]]
        X = torch.empty((m.ncol * L, 8, 3), dtype=torch.float64, device=like.device)
        for v in range(8):
            h = z[lev + v // 4]
            if m.geometry == 1:
                X[:, v] = corners[col, v % 4] * (m.radius + h)[:, None]
            else:
                X[:, v] = corners[col, v % 4]
                X[:, v, 2] = h

        def shape(x, y, w):
            ax, ay, aw = ((1 - x, x), (1 - y, y), (1 - w, w))
            n = [ax[v & 1] * ay[v >> 1 & 1] * aw[v >> 2] for v in range(8)]
            s = (-1.0, 1.0)
            d = [[s[v & 1] * ay[v >> 1 & 1] * aw[v >> 2], ax[v & 1] * s[v >> 1 & 1] * aw[v >> 2],
                  ax[v & 1] * ay[v >> 1 & 1] * s[v >> 2]] for v in range(8)]
            basis = [[0, y - 1, 0], [x, 0, 0], [0, y, 0], [x - 1, 0, 0], [0, 0, w - 1], [0, 0, w]]
            return [_t(np.array(a, np.float64), like) for a in (n, d, basis)]

        def up(x):
            if m.geometry == 1:
                return x / x.norm(dim=1, keepdim=True)
            r = torch.zeros_like(x)
            r[:, 2] = 1.0
            return r

        def mapped(x, y, w):
            n, d, basis = shape(x, y, w)
            J = X.transpose(1, 2) @ d
            V = J @ basis.T
            return torch.linalg.det(J), V, (up(torch.einsum("v,cvi->ci", n, X))[:, None] @ V)[:, 0]

        tl, el = f8(bg.theta_lev), f8(bg.exner_lev)
        dz, th0, th1 = z[lev + 1] - z[lev], tl[col, lev], tl[col, lev + 1]
        helm = co.preset == 1
        c22 = torch.zeros_like(dz) if helm else (-co.tau_u * co.tau_theta * co.dt ** 2 * co.cp *
                                                 (el[col, lev + 1] - el[col, lev]) / dz * (th1 - th0) / dz)
        cz = 0.0 if helm else co.tau_u * co.dt * 2 * co.omega
        gq = math.sqrt(15.0) / 10
        rule = [(0.5 - gq, 5 / 18), (0.5, 8 / 18), (0.5 + gq, 5 / 18)]
        M = torch.zeros((m.ncol * L, 6, 6), dtype=torch.float64, device=like.device)
        vol = torch.zeros_like(dz)
        for x, wx in rule:
            for y, wy in rule:
                for w, wz in rule:
                    det, V, rv = mapped(x, y, w)
                    q = V.transpose(1, 2) @ V + c22[:, None, None] * rv[:, :, None] * rv[:, None, :]
                    if cz:   # v_f . (c x v_g), c along the third axis
                        q += cz * (V[:, 1, :, None] * V[:, 0, None, :] - V[:, 0, :, None] * V[:, 1, None, :])
                    M += (wx * wy * wz / det)[:, None, None] * q
                    vol += wx * wy * wz * det
        vol1, _V, rvc = mapped(0.5, 0.5, 0.5)
        face = {}
        for e, ((a, b), (fa, fb)) in enumerate(zip(m.edge_cols.tolist(), m.edge_face.tolist())):
            face[a, fa], face[b, fb] = b, a
        nbr = i8([[face[c, f] for f in range(4)] for c in range(m.ncol)])
        theta = torch.empty((m.ncol * L, 6), dtype=torch.float64, device=like.device)
        mean = 0.5 * (tl[:, 1:] + tl[:, :-1])
        for f in range(4):
            theta[:, f] = 0.5 * (mean[col, lev] + mean[nbr[col, f], lev])
        theta[:, 4], theta[:, 5] = th0, th1
        if helm:
            kth, b, self.m = torch.ones_like(theta), torch.ones_like(theta), co.sigma * vol1
        else:
            kth = co.tau_u * co.dt * co.cp * theta
            b = (co.tau_rho * co.dt * vol1 / vol)[:, None] + (co.tau_theta * co.dt * (th1 - th0) / dz /
                                                              (0.5 * (th0 + th1)))[:, None] * rvc
            self.m = (1 - co.kappa) / co.kappa * vol1 / f8(bg.exner)[col, lev]
        d = M.diagonal(dim1=1, dim2=2).rsqrt()
        Mi = d[:, :, None] * torch.linalg.inv(d[:, :, None] * M * d[:, None, :]) * d[:, None, :]
        y, w = -(Mi @ kth[:, :, None])[:, :, 0], (Mi.transpose(1, 2) @ b[:, :, None])[:, :, 0]
        s = self.m - (b * y).sum(1)
        self.A = torch.cat([torch.cat([Mi + y[:, :, None] * w[:, None] / s[:, None, None], -(y / s[:, None])[:, :, None]], 2),
                            torch.cat([-w / s[:, None], 1 / s[:, None]], 1)[:, None]], 1)
        self.SK, self.kth, self.b = self.A[:, :6, :6] * kth[:, None, :], kth, b
        self.one = self.m[:, None] * -(y / s[:, None])          # S_K 1, as G annihilates constants
        self.lump = (M.diagonal(dim1=1, dim2=2).abs() +
                     torch.stack([M[:, f, o].abs() for f, o in enumerate((2, 3, 0, 1, 5, 4))], 1))
        first = _t(m.edge_cols[:, 0].astype(np.int64), like)
        ff = _t(m.edge_face[:, 0].astype(np.int64), like)
        fs = torch.arange(4, device=like.device)
        e = ce[col][:, :4]
        self.sign = torch.cat([torch.where((first[e] == col[:, None]) & (ff[e] == fs), 1.0, -1.0).double(),
                               torch.tensor([[-1.0, 1.0]], dtype=torch.float64, device=like.device).expand(len(col), 2)], 1)

    def add(self, v):
        out = torch.zeros(self.T, dtype=torch.float64, device=v.device)
        return out.index_add_(0, self.g.reshape(-1), v.reshape(-1))

    def S(self, x):
        return self.add((self.SK @ x[self.g][:, :, None])[:, :, 0])

    def rhs(self, R):
        return self.add((self.A @ R[:, :, None])[:, :6, 0])

    def weights(self):
        w = torch.full_like(self.kth, 0.5)
        w[:, 4][self.lev == 0] = 1.0
        w[:, 5][self.lev == self.L - 1] = 1.0
        return w

    def H(self, x):
        lump = self.add(self.lump)
        u = self.add(self.sign * -self.kth * x[:, None]) / lump
        inner = torch.ones(self.T, dtype=torch.bool, device=x.device)
        z = self.NH + torch.arange(self.ncol, device=x.device) * (self.L + 1)
        inner[z] = inner[z + self.L] = False
        return self.m * x - (self.sign * self.b * torch.where(inner, u, 0.0)[self.g]).sum(1)

    def sweep(self, b, x, omega=0.6):
        r = b - self.S(x)
        d = self.add(self.SK.diagonal(dim1=1, dim2=2))
        out = x.clone()
        out[:self.NH] += omega * r[:self.NH] / d[:self.NH]
        n, L = self.ncol, self.L
        dz, rz = d[self.NH:].view(n, L + 1), r[self.NH:].view(n, L + 1)
        up, lo = self.SK[:, 4, 5].view(n, L), self.SK[:, 5, 4].view(n, L)   # couplings k -> k + 1, k + 1 -> k
        c, y = [], []
        for k in range(L + 1):
            piv = dz[:, k] - (lo[:, k - 1] * c[k - 1] if k else 0.0)
            c.append(up[:, k] / piv if k < L else None)
            y.append((rz[:, k] - (lo[:, k - 1] * y[k - 1] if k else 0.0)) / piv)
        for k in range(L - 1, -1, -1):
            y[k] = y[k] - c[k] * y[k + 1]
        out[self.NH:] += omega * torch.stack(y, 1).reshape(-1)
        return out


class _Boxes:
    """Degree p on the uniform plane: every cell is the same box, with Kronecker-product blocks."""

    def __init__(self, case, like):
        hier, co = _of(case)
        m, p = hier.meshes[0], case["degree"]
        nt, L = p + 1, m.nlev
        xg, wg = np.polynomial.legendre.leggauss(nt)
        xg, wg = 0.5 * (xg + 1), 0.5 * wg
        inner = np.sort(np.polynomial.legendre.Legendre.basis(p + 1).deriv().roots().real)
        xl = 0.5 * (np.concatenate([[-1.0], inner, [1.0]]) + 1)
        qx, qw = np.polynomial.legendre.leggauss(p + 3)
        qx, qw = 0.5 * (qx + 1), 0.5 * qw
        poly = lambda nodes: [np.polynomial.Polynomial.fromroots(np.delete(nodes, i)) /
                              np.prod(nodes[i] - np.delete(nodes, i)) for i in range(len(nodes))]
        NL, GL = poly(xl), poly(xg)
        mass = np.array([[np.sum(qw * a(qx) * b(qx)) for b in NL] for a in NL])
        diff = np.array([[np.sum(qw * a.deriv()(qx) * b(qx)) for b in GL] for a in NL])
        h = np.array([1.0 / m.n_per_side] * 2 + [0.1 / L])
        det = h.prod()
        comp, far, sgn = (1, 0, 1, 0, 2, 2), (0, 1, 1, 0, 0, 1), (-1, 1, 1, -1, -1, 1)
        dofs = [(comp[f], far[f] * (p + 1), p - s if f in (2, 3) else s, t, sgn[f])
                for f in range(6) for s in range(nt) for t in range(nt)]
        dofs += [(d, a, b, c, 1) for d in range(3) for a in range(1, p + 1) for b in range(nt) for c in range(nt)]
        nu, npr, nb = len(dofs), nt ** 3, nt * nt
        A = np.zeros((nu + npr, nu + npr))
        for i, (d, a, b, c, s) in enumerate(dofs):
            for j, (d2, a2, b2, c2, s2) in enumerate(dofs):
                if (d, b, c) == (d2, b2, c2):
                    A[i, j] = s * s2 * h[d] ** 2 / det * mass[a, a2] * wg[b] * wg[c]
            for k in range(nt):
                at = [b, c]
                at.insert(d, k)
                j = nu + (at[0] * nt + at[1]) * nt + at[2]
                A[i, j] = -s * diff[a, k] * wg[b] * wg[c]
                A[j, i] = -A[i, j]
        for j in range(npr):
            A[nu + j, nu + j] = co.sigma * det * wg[j // nb] * wg[j // nt % nt] * wg[j % nt]
        e = 1 / np.sqrt(np.abs(np.diag(A)))
        self.A = _t(e[:, None] * np.linalg.inv(e[:, None] * A * e) * e, like)
        self.C = _t(np.tile(np.outer(wg, wg).ravel(), 6), like)
        self.m = co.sigma * det
        col, lev = np.divmod(np.arange(m.ncol * L), L)
        g = np.zeros((m.ncol * L, 6, nt, nt), np.int64)
        st = np.arange(nt)
        for f in range(4):
            ed = m.col_edges[col, f].astype(np.int64)
            own = (m.edge_cols[ed, 0] == col) & (m.edge_face[ed, 0] == f)
            s = np.where(own[:, None], st, p - st)
            g[:, f] = nb * (ed * L + lev)[:, None, None] + nt * s[:, :, None] + st
        for f in (4, 5):
            g[:, f] = nb * (m.nedge * L + col * (L + 1) + lev + f - 4)[:, None, None] + nt * st[:, None] + st
        self.g = _t(g.reshape(len(col), -1), like)
        self.T, self.nf, self.nu, self.nb = nb * (m.nedge * L + m.ncol * (L + 1)), 6 * nb, nu, nb
        self.lev, self.L = _t(lev, like), L

    def add(self, v):
        out = torch.zeros(self.T, dtype=torch.float64, device=v.device)
        return out.index_add_(0, self.g.reshape(-1), v.reshape(-1))

    def S(self, x):
        return self.add((self.C * x[self.g]) @ self.A[:self.nf, :self.nf].T * self.C)

    def rhs(self, R):
        return self.add((R @ self.A.T)[:, :self.nf] * self.C)

    def recover(self, lam, R):
        R = R.clone()
        R[:, :self.nf] -= self.C * lam[self.g]
        X = R @ self.A.T
        return X[:, :self.nu].reshape(-1), X[:, self.nu:].reshape(-1)

    def gamma(self):
        s1 = self.S(torch.ones(self.T, dtype=torch.float64, device=self.C.device))[self.g].view(-1, 6, self.nb).sum(2)
        w = torch.full_like(s1, 0.5)
        w[:, 4][self.lev == 0] = 1.0
        w[:, 5][self.lev == self.L - 1] = 1.0
        return self.m / (w * s1).sum(1)


def _network(case, seed):
    """Loss and gradient of the coarse map with BF16-stored weights and activations."""
    x, t, w = _patches(case, seed)
    x, t = x.double(), t.double()
    W = {k: _t(v, x).requires_grad_() for k, v in I.unflatten_coarse_model(w).items()}
    q = lambda a: a + (a.detach().to(torch.bfloat16).double() - a.detach())   # straight through
    n, nx, ny, L = case["nsamp"], case["nx"], case["ny"], case["nlev"]
    conv = lambda k, v: torch.nn.functional.conv1d(v, q(W[k]), padding=1)
    h = q(conv("W2", q(conv("W1", q(x).view(-1, 1, L)).relu())).relu())
    ch = h.shape[1]
    hp = torch.nn.functional.pad(h.view(n, ny, nx, ch, L).permute(0, 3, 4, 1, 2), (1, 1, 1, 1))
    at = lambda i, j: hp[..., 1 + j:1 + j + ny, 1 + i:1 + i + nx]
    edge = at(1, 0) + at(-1, 0) + at(0, 1) + at(0, -1)
    diag = at(1, 1) + at(-1, 1) + at(1, -1) + at(-1, -1)
    mix = q(W["M"])[None, :, :, None, None, None]
    h3 = q((mix[:, :, 0] * at(0, 0) + mix[:, :, 1] * edge + mix[:, :, 2] * diag).relu())
    y = conv("W3", h3.permute(0, 3, 4, 1, 2).reshape(-1, ch, L)).view(n, nx * ny, L)
    loss = (((y - t) ** 2).sum((1, 2)) / (t ** 2).sum((1, 2))).mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grad": torch.cat([W[k].grad.reshape(-1) for k in ("W1", "W2", "M", "W3")])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None
    if kind == "grad":
        return _network(case, seed)
    C, T, nu, npr = _sizes(case)
    if kind == "solve" and T > 8000:   # a dense solve is out of reach
        return None
    Ru, Rp, x, b, c = _data(case, seed)
    R = torch.cat([Ru.view(C, nu), Rp.view(C, npr)], 1)
    e = (_Cells if case["degree"] == 0 else _Boxes)(case, x)
    if kind == "apply":
        return e.S(x)
    if kind == "smooth":
        for _ in range(case["sweeps"]):
            x = e.sweep(b, x)
        return x
    if kind == "setup":
        out = {"B": e.rhs(R), "Sx": e.S(x)}
        if case["degree"] == 0:
            return dict(out, gamma=e.m / (e.weights() * e.add(e.one)[e.g]).sum(1), Hc=e.H(c))
        out["u"], out["pi"] = e.recover(x, R)
        return dict(out, gamma=e.gamma())
    n = e.g.shape[1]
    SK = e.SK if case["degree"] == 0 else (e.C[:, None] * e.A[:n, :n] * e.C).expand(C, n, n)
    S = torch.zeros((T, T), dtype=torch.float64, device=x.device)
    S.view(-1).index_add_(0, (e.g[:, :, None] * T + e.g[:, None, :]).reshape(-1), SK.reshape(-1))
    lam = torch.linalg.solve(S, e.rhs(R))
    if case["degree"] == 0:
        R[:, :6] -= e.kth * lam[e.g]
        X = (e.A @ R[:, :, None])[:, :, 0]
        return {"lam": lam, "u": X[:, :6].reshape(-1), "pi": X[:, 6]}
    u, pi = e.recover(lam, R)
    return {"lam": lam, "u": u, "pi": pi}

"""The work a user of the solver has it do, as cases to be timed and checked.

Every case goes through the public Python entry points (helmholtz_apply, mg_smooth, vcycle,
pressure_solve, solve, mixed_solve, solve_mixed, Ensemble).  Sizes are those of the repository's
own workloads (C12L30 up to C192L70, 30 / 50 / 70 levels, the uneven ensemble) and of its tests
(odd and ragged meshes, odd level counts).  ``exact`` restates each result in plain torch FP64: its
own cubed-sphere geometry, couplings, line smoother, V-cycle and Krylov solve.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2002_00756_gb300 as mg

RADIUS, CS, DT, TOP = 6371.0e3, 340.0, 600.0, 30.0e3
OMEGA, N_PRE, N_POST, N_COARSE, RESTART = 0.8, 2, 2, 4, 5
EPS = 0.05                      # strength of the mixed system's vertical buoyancy coupling
ROTATION = 7.292e-5             # the Earth's angular velocity, for the implicit Coriolis term
EXACT_TOL = 1e-13               # relative residual of the FP64 reference solves

DEV = "cuda"


def listed():
    return [
        # smallest call: one operator apply on the coarsest mesh a test or a tutorial uses
        {"name": "apply_c12l30", "kind": "apply", "n": 12, "nlev": 30, "levels": 3, "precision": "fp64"},
        # a small solve in the plain method: launch latency counts
        {"name": "solve_c12l30_fp64", "kind": "solve", "n": 12, "nlev": 30, "levels": 3, "precision": "fp64",
         "tol": 1e-8},
        # line smoothing as a building block, on an odd mesh with an odd number of levels
        {"name": "smooth_c45l37", "kind": "smooth", "n": 45, "nlev": 37, "levels": 1, "precision": "fp64",
         "sweeps": 3},
        # the V-cycle as the preconditioner of a caller's own FP64 Krylov method
        {"name": "vcycle_c96l70_fp64", "kind": "vcycle", "n": 96, "nlev": 70, "levels": 4, "precision": "fp64"},
        # an ordinary pressure solve with the FP32 V-cycle
        {"name": "solve_c48l30_fp32", "kind": "solve", "n": 48, "nlev": 30, "levels": 4, "precision": "fp32",
         "tol": 1e-8},
        # BF16 coefficients on a mesh with ragged blocks and an odd number of levels
        {"name": "solve_c90l41_bf16", "kind": "solve", "n": 90, "nlev": 41, "levels": 2, "precision": "fp32_bf16",
         "tol": 1e-8},
        # FP32 V-cycle with the finest level's column elimination in FP64
        {"name": "solve_c96l70_p64", "kind": "solve", "n": 96, "nlev": 70, "levels": 4, "precision": "fp32_p64",
         "tol": 1e-8},
        # the benchmarked solve, the largest workload of the repository
        {"name": "solve_c192l70_fp32", "kind": "solve", "n": 192, "nlev": 70, "levels": 4, "precision": "fp32",
         "tol": 2e-9},
        # differentiable solve with the couplings as an input: forward, adjoint, both gradients
        {"name": "grad_c96l70_fp32", "kind": "grad", "n": 96, "nlev": 70, "levels": 4, "precision": "fp32",
         "tol": 1e-8},
        # the full mixed (velocity, pressure) system
        {"name": "mixed_c48l30_fp32", "kind": "mixed", "n": 48, "nlev": 30, "levels": 4, "precision": "fp32",
         "tol": 1e-8, "consistent": False},
        # differentiable mixed solve with the consistent mass and the Coriolis term
        {"name": "mixed_grad_c48l30_fp32", "kind": "mixed_grad", "n": 48, "nlev": 30, "levels": 4,
         "precision": "fp32", "tol": 1e-8, "consistent": True},
        # uneven ensemble members in one graph launch
        {"name": "ensemble_12_fp32", "kind": "ensemble", "members": 12, "pick": 20020, "precision": "fp32",
         "tol": 1e-8},
    ]


def draw(rng):
    def size(lo, hi, levels):
        q = 1 << (levels - 1)
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return max(q, n // q * q)

    kind = rng.choice(["apply", "smooth", "vcycle", "solve", "solve", "solve", "grad", "mixed", "mixed_grad",
                       "ensemble"])
    levels = rng.choice([2, 3, 4])
    nlev = int(round(math.exp(rng.uniform(math.log(10), math.log(80)))))
    case = {"kind": kind, "levels": levels, "nlev": nlev}
    if kind == "apply":
        return {**case, "n": size(12, 160, levels), "precision": "fp64"}
    if kind == "smooth":
        case["levels"] = 1
        return {**case, "n": size(9, 120, 1), "precision": "fp64", "sweeps": rng.randint(1, 4)}
    if kind == "vcycle":
        return {**case, "n": size(12, 128, levels), "precision": "fp64"}
    if kind == "solve":
        prec = rng.choice(["fp64", "fp32", "fp32", "fp32_p64", "fp32_bf16"])
        return {**case, "n": size(12, 160 if prec == "fp32" else 112, levels), "precision": prec,
                "tol": rng.choice([1e-6, 1e-8, 2e-9])}
    if kind == "grad":
        return {**case, "n": size(12, 96, levels), "precision": rng.choice(["fp32", "fp64"]), "tol": 1e-8}
    if kind in ("mixed", "mixed_grad"):
        return {**case, "n": size(12, 64, levels), "precision": rng.choice(["fp32", "fp64"]), "tol": 1e-8,
                "consistent": rng.choice([False, True])}
    return {"kind": kind, "members": rng.randint(4, 12), "pick": rng.randrange(1 << 20), "precision": "fp32",
            "tol": 1e-8}


def _members(case):
    """(n, nlev) of an ensemble's members: the uneven sizes of the repository's ensemble."""
    r = random.Random(case["pick"])
    return [(r.choice([32, 48, 64, 96]), r.choice([30, 50, 70])) for _ in range(case["members"])]


# ---- inputs ----------------------------------------------------------------------------

def _heights(nlev):
    s, beta = np.arange(nlev + 1) / nlev, 5.0 / 29.0
    return TOP * (beta * s + (1.0 - beta) * s * s)


def _rand(seed, stream, count, kind="normal"):
    g = torch.Generator(device=DEV).manual_seed((seed * 1009 + stream) % (1 << 62))
    f = torch.randn if kind == "normal" else torch.rand
    return f(count, generator=g, device=DEV, dtype=torch.float64)


def _factors(seed, nlev, ncol):
    """Lognormal(0, 0.1) background-state factors, one per cell."""
    return torch.exp(0.1 * _rand(seed, 1, nlev * ncol)).view(nlev, ncol)


def _mixed_inputs(seed, nlev, ncol):
    nh, nv = 2 * ncol * nlev, ncol * (nlev + 1)
    bu, bd = (_rand(seed, s, nv, "uniform").view(nlev + 1, ncol) for s in (3, 4))
    ru = _rand(seed, 5, nh + nv)
    ru[nh:nh + ncol] = 0.0          # no flux through surface and lid
    ru[nh + nv - ncol:] = 0.0
    return bu, bd, ru, _rand(seed, 6, nlev * ncol)


def _f0(case):
    return 0.5 * DT * 2.0 * ROTATION if case["consistent"] else 0.0


def _handle(n, nlev, levels, precision, g, **kw):
    return mg.mg_setup(n, nlev, _heights(nlev), g.cpu().numpy(), radius=RADIUS, cs_dt=CS * DT, levels=levels,
                       omega=OMEGA, n_pre=N_PRE, n_post=N_POST, n_coarse=N_COARSE, precision=precision,
                       gcr_restart=RESTART, **kw)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        hs, bs = [], []
        for i, (n, nlev) in enumerate(_members(case)):
            g = _factors(seed + 7919 * (i + 1), nlev, 6 * n * n)
            hs.append(_handle(n, nlev, 4, case["precision"], g))
            bs.append(_rand(seed + 7919 * (i + 1), 2, g.numel()))
        xs = [torch.zeros_like(b) for b in bs]
        return {"kind": kind, "xs": xs, "ens": mg.Ensemble(hs, bs, xs, tol=case["tol"])}
    n, nlev = case["n"], case["nlev"]
    ncol = 6 * n * n
    g = _factors(seed, nlev, ncol)
    s = {"kind": kind, "tol": case.get("tol"), "sweeps": case.get("sweeps")}
    if kind in ("mixed", "mixed_grad"):
        bu, bd, ru, rp = _mixed_inputs(seed, nlev, ncol)
        s["h"] = _handle(n, nlev, case["levels"], case["precision"], g, beta_up=bu.cpu().numpy(),
                         beta_dn=bd.cpu().numpy(), eps=EPS, consistent_mass=case["consistent"],
                         coriolis_f0=_f0(case))
        s |= {"ru": ru, "rp": rp, "u": torch.zeros_like(ru), "p": torch.zeros_like(rp)}
        if kind == "mixed_grad":
            s |= {"wu": torch.exp(0.5 * _rand(seed, 8, ru.numel())), "wp": torch.exp(0.5 * _rand(seed, 9, rp.numel()))}
            ru.requires_grad_(True)
            rp.requires_grad_(True)
        return s
    s["h"] = _handle(n, nlev, case["levels"], case["precision"], g)
    s["b"] = _rand(seed, 2, nlev * ncol)
    s["x"] = torch.zeros_like(s["b"])
    if kind == "smooth":
        s["x0"] = _rand(seed, 7, nlev * ncol)
    if kind == "grad":
        s["w"] = torch.exp(0.5 * _rand(seed, 8, nlev * ncol))
        s["a"] = _couplings(_mesh(n), nlev, g).reshape(-1).contiguous().requires_grad_(True)
        s["b"].requires_grad_(True)
    return s


def run(state):
    kind = state["kind"]
    if kind == "ensemble":
        state["ens"].solve()
        return state["xs"]
    h = state["h"]
    if kind == "apply":
        mg.helmholtz_apply(h, state["b"], state["x"])
        return state["x"]
    if kind == "smooth":
        mg.mg_smooth(h, 0, state["b"], state["x0"], state["x"], state["sweeps"])
        return state["x"]
    if kind == "vcycle":
        mg.vcycle(h, state["b"], state["x"])
        return state["x"]
    if kind == "solve":
        mg.pressure_solve(h, state["b"], state["x"], tol=state["tol"])
        return state["x"]
    if kind == "grad":
        x = mg.solve(h, state["b"], tol=state["tol"], coeffs=state["a"])
        loss = 0.5 * ((state["w"] * x) ** 2).sum()
        gb, ga = torch.autograd.grad(loss, (state["b"], state["a"]))
        return {"x": x.detach(), "db": gb, "da": ga}
    if kind == "mixed":
        mg.mixed_solve(h, state["ru"], state["rp"], state["u"], state["p"], tol=state["tol"])
        return {"u": state["u"], "p": state["p"]}
    u, p = mg.solve_mixed(h, state["ru"], state["rp"], tol=state["tol"])
    loss = 0.5 * ((state["wu"] * u) ** 2).sum() + 0.5 * ((state["wp"] * p) ** 2).sum()
    gu, gp = torch.autograd.grad(loss, (state["ru"], state["rp"]))
    return {"u": u.detach(), "p": p.detach(), "du": gu, "dp": gp}


def work(case):
    """Inputs read once and outputs written once; operations of the sweeps, transfers and Krylov
    steps the method itself takes (about 8 iterations to 1e-8 on these operators)."""
    kind = case["kind"]
    if kind == "ensemble":
        cells = sum(6 * n * n * nlev for n, nlev in _members(case))
        return {"bytes": 8.0 * cells * 5, "flops": cells * 8 * 230.0}
    cells = float(6 * case["n"] ** 2 * case["nlev"])
    sweep, cyc = 25.0, (N_PRE + N_POST) * 25.0 * 4 / 3 + 20.0     # flops per cell
    if kind == "apply":
        return {"bytes": 8.0 * cells * 5, "flops": 18.0 * cells}          # x, y, 3 face couplings
    if kind == "smooth":
        return {"bytes": 8.0 * cells * 6, "flops": case["sweeps"] * sweep * cells}
    if kind == "vcycle":
        return {"bytes": 8.0 * cells * 5, "flops": cyc * cells}
    its = 6 if case["tol"] >= 1e-6 else 8 if case["tol"] >= 1e-8 else 10
    solve = its * (cyc + 60.0) * cells
    if kind == "solve":
        return {"bytes": 8.0 * cells * 5, "flops": solve}
    if kind == "grad":                                                     # b, w, x, db; a and da
        return {"bytes": 8.0 * cells * (4 + 12), "flops": 2 * solve}
    mixed = its * (cyc + 200.0) * cells
    if kind == "mixed":
        return {"bytes": 8.0 * cells * (4 + 4 + 8), "flops": mixed}        # rhs, solution, operator
    return {"bytes": 8.0 * cells * (8 + 8 + 8), "flops": 2 * mixed}


# ---- the results in plain FP64 ----------------------------------------------------------
# Equiangular gnomonic cubed sphere, strong lowest-order operator
#   (H x)_i = x_i + sum_f a_if (x_i - x_j),  a_if = (c_s dt)^2 g_f mu_f A_f / (V_i d_f),
# sides E, W, N, S, up, down; fields are (nlev, ncol).

_meshes = {}


def _mesh(n):
    if n not in _meshes:
        d, q = 0.5 * math.pi / n, 0.25 * math.pi
        p, j, i = (v.ravel() for v in np.meshgrid(np.arange(6), np.arange(n), np.arange(n), indexing="ij"))

        def sphere(xi, eta):
            a, b, o = np.tan(xi), np.tan(eta), np.ones_like(xi)
            v = np.choose(p, [np.stack(t) for t in ((o, a, b), (-a, o, b), (-o, -a, b), (a, -o, b), (-b, a, o),
                                                      (b, a, -o))])
            return v / np.linalg.norm(v, axis=0)

        def arc(u, v):
            return np.arctan2(np.linalg.norm(np.cross(u, v, axis=0), axis=0), (u * v).sum(0))

        def cell(v):
            x, y, z = v
            ax, ay, az = np.abs(v)
            fx, fy = (ax >= ay) & (ax >= az), (ay >= az)
            pn = np.where(fx, np.where(x > 0, 0, 2), np.where(fy, np.where(y > 0, 1, 3), np.where(z > 0, 4, 5)))
            a = np.choose(pn, [y / x, -x / y, y / x, -x / y, y / z, -y / z])
            b = np.choose(pn, [z / x, z / y, -z / x, -z / y, -x / z, -x / z])
            at = [np.clip(np.floor((np.arctan(t) + q) / d).astype(np.int64), 0, n - 1) for t in (a, b)]
            return pn * n * n + at[1] * n + at[0]

        x0, y0 = -q + d * i, -q + d * j
        c00, c10, c11, c01 = sphere(x0, y0), sphere(x0 + d, y0), sphere(x0 + d, y0 + d), sphere(x0, y0 + d)
        mid = sphere(x0 + 0.5 * d, y0 + 0.5 * d)
        F = lambda x, y: np.arctan(x * y / np.sqrt(1.0 + x * x + y * y))  # noqa: E731
        t = np.tan
        area = RADIUS ** 2 * (F(t(x0 + d), t(y0 + d)) - F(t(x0), t(y0 + d)) - F(t(x0 + d), t(y0)) + F(t(x0), t(y0)))
        with np.errstate(divide="ignore", invalid="ignore"):
            nbr = np.stack([cell(sphere(x0 + (0.5 + 0.75 * u) * d, y0 + (0.5 + 0.75 * v) * d))
                            for u, v in ((1, 0), (-1, 0), (0, 1), (0, -1))])
        own = np.arange(6 * n * n)
        side = np.stack([np.argmax(nbr[:, nbr[s]] == own, axis=0) for s in range(4)])
        edge = RADIUS * np.stack([arc(c10, c11), arc(c00, c01), arc(c01, c11), arc(c00, c10)])
        dist = RADIUS * np.stack([arc(mid, mid[:, nbr[s]]) for s in range(4)])
        owner, sd = np.nonzero((own < nbr).T)      # faces under their lower column, by (column, side)
        fof = np.zeros((4, 6 * n * n), np.int64)
        fof[sd, owner] = np.arange(owner.size)
        fof[side[sd, owner], nbr[sd, owner]] = np.arange(owner.size)
        T = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(DEV)  # noqa: E731
        m = {"n": n, "ncol": 6 * n * n, "nbr": T(nbr), "side": T(side), "area": T(area), "edge": T(edge),
             "dist": T(dist), "sinlat": T(mid[2]), "faceL": T(owner), "faceR": T(nbr[sd, owner]), "faceS": T(sd),
             "fof": T(fof)}
        if n % 2 == 0:
            nc = n // 2
            m["parent"] = T(p * nc * nc + (j // 2) * nc + i // 2)
        _meshes[n] = m
    return _meshes[n]


def _vertical(nlev):
    z = torch.from_numpy(_heights(nlev)).to(DEV)
    dz = z[1:] - z[:-1]
    dzc = torch.ones(nlev + 1, device=DEV, dtype=torch.float64)
    dzc[1:-1] = 0.5 * (z[2:] - z[:-2])
    return dz, dzc


def _couplings(m, nlev, g, mu=None, muh=None):
    dz, dzc = _vertical(nlev)
    c2 = (CS * DT) ** 2
    a = torch.zeros(6, nlev, m["ncol"], device=DEV, dtype=torch.float64)
    for s in range(4):
        geo = m["edge"][s] / (m["dist"][s] * m["area"])
        if muh is not None:
            geo = geo * muh[m["fof"][s]]
        a[s] = c2 * 0.5 * (g + g[:, m["nbr"][s]]) * geo
    flux = c2 * 0.5 * (g[1:] + g[:-1]) / dzc[1:-1, None]
    if mu is not None:
        flux = flux * mu[1:-1]
    a[4, :-1] = flux / dz[:-1, None]
    a[5, 1:] = flux / dz[1:, None]
    # one value per face: V_i a_if = V_j a_jf to the last bit, as a caller's face-based code gives it
    v = m["area"]
    fv = torch.empty(nlev, 2 * m["ncol"], device=DEV, dtype=torch.float64)
    fv[:] = a[m["faceS"], :, m["faceL"]].T * v[m["faceL"]]
    for s in range(4):
        a[s] = fv[:, m["fof"][s]] / v
    return a


def _apply(m, a, x):
    y = x.clone()
    for s in range(4):
        y += a[s] * (x - x[:, m["nbr"][s]])
    y[:-1] += a[4, :-1] * (x[:-1] - x[1:])
    y[1:] += a[5, 1:] * (x[1:] - x[:-1])
    return y


class _Level:
    def __init__(self, m, a):
        self.m, self.a = m, a
        nlev = a.shape[1]
        s = 1.0 + a[:4].sum(0)
        self.mul, self.ip, self.e = torch.zeros_like(s), torch.empty_like(s), torch.empty_like(s)
        q = s[0]
        for k in range(nlev):      # pivots as sums of positive terms
            if k:
                self.mul[k] = a[5, k] * self.ip[k - 1]
                q = s[k] + self.mul[k] * q
            self.ip[k] = 1.0 / (q + a[4, k])
            self.e[k] = a[4, k] * self.ip[k]

    def sweep(self, b, x):
        r = b if x is None else b - _apply(self.m, self.a, x)
        y = torch.empty_like(r)
        y[0] = r[0]
        for k in range(1, r.shape[0]):
            torch.addcmul(r[k], self.mul[k], y[k - 1], out=y[k])
        y *= self.ip
        for k in range(r.shape[0] - 2, -1, -1):
            y[k].addcmul_(self.e[k], y[k + 1])
        return OMEGA * y if x is None else x + OMEGA * y


def _hierarchy(n, nlev, levels, g, mu=None, muh=None):
    out = []
    for l in range(levels):
        m = _mesh(n >> l)
        out.append(_Level(m, _couplings(m, nlev, g, mu, muh)))
        if l + 1 < levels:
            mean = lambda f, c=_mesh(n >> (l + 1)), m=m: torch.zeros(  # noqa: E731
                f.shape[0], c["ncol"], device=DEV, dtype=torch.float64).index_add_(1, m["parent"], f * m["area"]) / c["area"]
            g = mean(g)
            mu = None if mu is None else mean(mu)
            if muh is not None:       # edge-length-weighted mean of a coarse face's two fine faces
                c = _mesh(n >> (l + 1))
                num, den = (torch.zeros(2 * c["ncol"], device=DEV, dtype=torch.float64) for _ in range(2))
                for s in range(4):
                    par = m["parent"]
                    # fine cells whose neighbour across s has another parent lie on the coarse face
                    on = par[m["nbr"][s]] != par
                    F, f = c["fof"][s][par[on]], m["fof"][s][on]
                    own = m["faceL"][f] == torch.nonzero(on)[:, 0]
                    w = m["edge"][s][on] * own
                    num.index_add_(0, F, w * muh[f])
                    den.index_add_(0, F, w)
                muh = num / den
    return out


def _vcycle(lv, b, l=0):
    L, x = lv[l], None
    if l == len(lv) - 1:
        for _ in range(N_COARSE):
            x = L.sweep(b, x)
        return x
    for _ in range(N_PRE):
        x = L.sweep(b, x)
    r = b if x is None else b - _apply(L.m, L.a, x)
    c = lv[l + 1].m
    bc = torch.zeros(b.shape[0], c["ncol"], device=DEV, dtype=torch.float64)
    bc.index_add_(1, L.m["parent"], r * L.m["area"])
    x = x + _vcycle(lv, bc / c["area"], l + 1)[:, L.m["parent"]]
    for _ in range(N_POST):
        x = L.sweep(b, x)
    return x


def _krylov(A, P, b):
    """GCR with every direction kept, to a relative residual of EXACT_TOL (recursive)."""
    x, r, zs, ws = torch.zeros_like(b), b.clone(), [], []
    bn = b.norm()
    for _ in range(80):
        if r.norm() <= EXACT_TOL * bn:
            break
        z = P(r)
        w = A(z)
        for zi, wi in zip(zs, ws):
            c = torch.dot(w, wi)
            w.sub_(wi, alpha=float(c))
            z.sub_(zi, alpha=float(c))
        s = w.norm()
        w, z = w / s, z / s
        zs.append(z)
        ws.append(w)
        c = float(torch.dot(r, w))
        x.add_(z, alpha=c)
        r.sub_(w, alpha=c)
    return x


def _solve_h(lv, b):
    shape = lv[0].a.shape[1:]
    return _krylov(lambda v: _apply(lv[0].m, lv[0].a, v.view(shape)).view(-1), lambda v: _vcycle(lv, v.view(shape)).view(-1), b)


class _Mixed:
    """[u; p] rows: M u + kd (p_R - p_L) = r_u, p + D u = r_p; M = velocity mass with the
    vertical buoyancy coupling and, optionally, the consistent mass and the Coriolis term."""

    def __init__(self, n, nlev, levels, g, bu, bd, consistent, f0):
        m = self.m = _mesh(n)
        self.nlev, self.ncol, self.nh = nlev, m["ncol"], 2 * m["ncol"] * nlev
        dz, dzc = _vertical(nlev)
        c = CS * DT
        L, R, S = m["faceL"], m["faceR"], m["faceS"]
        self.L, self.R = L, R
        self.kdh = c * 0.5 * (g[:, L] + g[:, R]) / m["dist"][S, L]
        self.kdv = torch.zeros(nlev + 1, self.ncol, device=DEV, dtype=torch.float64)
        self.kdv[1:-1] = c * 0.5 * (g[1:] + g[:-1]) / dzc[1:-1, None]
        len_ = m["edge"][S, L]
        self.dL, self.dR, self.dv = c * len_ / m["area"][L], c * len_ / m["area"][R], (c / dz)[:, None]
        # horizontal mass: triples (row face, column face, weight), the same on every level
        rows, cols, vals = [], [], []
        lump = torch.zeros(2 * self.ncol, device=DEV, dtype=torch.float64)
        own = torch.arange(self.ncol, device=DEV)
        F = f0 * m["sinlat"]
        out = (1.0, -1.0, 1.0, -1.0)
        tau = [out[s] * torch.where(L[m["fof"][s]] == own, 1.0, -1.0).double() for s in range(4)]
        for s in range(4):
            lump.index_add_(0, m["fof"][s], 0.5 + (-0.5 if s < 2 else 0.5) * F)
            for t in range(4):
                if t == s:
                    w = torch.full_like(F, 1.0 / 3.0 if consistent else 0.5)
                elif t == s ^ 1:
                    w = torch.full_like(F, 1.0 / 6.0 if consistent else 0.0)
                else:
                    w = F * (-0.25 if s < 2 else 0.25)
                rows.append(m["fof"][s])
                cols.append(m["fof"][t])
                vals.append(tau[s] * tau[t] * w)
        self.rows, self.cols, self.vals = torch.cat(rows), torch.cat(cols), torch.cat(vals)
        off, self.mv = (1.0 / 6.0, 2.0 / 3.0) if consistent else (0.0, 1.0)
        self.up, self.dn = torch.zeros_like(self.kdv), torch.zeros_like(self.kdv)
        self.up[1:nlev - 1] = EPS * bu[1:nlev - 1] + off
        self.dn[2:nlev] = EPS * bd[2:nlev] + off
        lv = self.mv + self.up + self.dn
        lv[0] = lv[-1] = 1.0
        self.rmh, self.rmv = 1.0 / lump, 1.0 / lv
        self.lv = _hierarchy(n, nlev, levels, g, self.rmv, self.rmh)
        # weights under which A^T = S J (A with the transposed mass) J S^-1
        gf = 0.5 * (g[:, L] + g[:, R])
        self.Wh = len_ * m["dist"][S, L] * dz[:, None] / gf
        self.Wv = torch.empty_like(self.kdv)
        self.Wv[1:-1] = m["area"] * dzc[1:-1, None] / (0.5 * (g[1:] + g[:-1]))
        self.Wv[0], self.Wv[-1] = m["area"] * dz[0] / g[0], m["area"] * dz[-1] / g[-1]
        self.V = m["area"] * dz[:, None]

    def split(self, v):
        nv = (self.nlev + 1) * self.ncol
        return (v[:self.nh].view(self.nlev, -1), v[self.nh:self.nh + nv].view(self.nlev + 1, -1),
                v[self.nh + nv:].view(self.nlev, -1))

    def div(self, uh, uv):
        y = torch.zeros(self.nlev, self.ncol, device=DEV, dtype=torch.float64)
        y.index_add_(1, self.L, uh * self.dL)
        y.index_add_(1, self.R, -uh * self.dR)
        y[:-1] += self.dv[:-1] * uv[1:-1]
        y[1:] -= self.dv[1:] * uv[1:-1]
        return y

    def grad(self, p):
        gv = torch.zeros_like(self.kdv)
        gv[1:-1] = self.kdv[1:-1] * (p[1:] - p[:-1])
        return self.kdh * (p[:, self.R] - p[:, self.L]), gv

    def mass(self, uh, uv, transpose=False):
        r, c = (self.cols, self.rows) if transpose else (self.rows, self.cols)
        yh = torch.zeros_like(uh).index_add_(1, r, uh[:, c] * self.vals)
        yv = uv.clone()
        yv[1:-1] = self.mv * uv[1:-1]
        if transpose:
            yv[2:-1] += self.up[1:-2] * uv[1:-2]
            yv[1:-2] += self.dn[2:-1] * uv[2:-1]
        else:
            yv[1:-1] += self.up[1:-1] * uv[2:] + self.dn[1:-1] * uv[:-2]
        return yh, yv

    def apply(self, v):
        uh, uv, p = self.split(v)
        (mh, mv), (gh, gv) = self.mass(uh, uv), self.grad(p)
        return torch.cat([(mh + gh).view(-1), (mv + gv).view(-1), (p + self.div(uh, uv)).view(-1)])

    def apply_t(self, v):
        """A^T v: M^T u + D^T p and G^T u + p."""
        uh, uv, p = self.split(v)
        mh, mv = self.mass(uh, uv, transpose=True)
        q = self.dv * p
        mh = mh + p[:, self.L] * self.dL - p[:, self.R] * self.dR
        mv[1:-1] += q[:-1] - q[1:]
        y = p.clone()
        t = self.kdh * uh
        y.index_add_(1, self.R, t)
        y.index_add_(1, self.L, -t)
        t = self.kdv[1:-1] * uv[1:-1]
        y[1:] += t
        y[:-1] -= t
        return torch.cat([mh.reshape(-1), mv.view(-1), y.view(-1)])

    def precond(self, v):
        uh, uv, p = self.split(v)
        b = p - self.div(uh * self.rmh, uv * self.rmv)
        p = _vcycle(self.lv, b)
        gh, gv = self.grad(p)
        return torch.cat([((uh - gh) * self.rmh).view(-1), ((uv - gv) * self.rmv).view(-1), p.reshape(-1)])

    def precond_t(self, v):
        S = torch.cat([self.Wh.view(-1), self.Wv.view(-1), -self.V.reshape(-1)])
        return S * self.precond(v / S)


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        xs = []
        for i, (n, nlev) in enumerate(_members(case)):
            s = seed + 7919 * (i + 1)
            g = _factors(s, nlev, 6 * n * n)
            xs.append(_solve_h(_hierarchy(n, nlev, 4, g), _rand(s, 2, g.numel())))
        return xs
    n, nlev = case["n"], case["nlev"]
    ncol = 6 * n * n
    g = _factors(seed, nlev, ncol)
    if kind in ("mixed", "mixed_grad"):
        bu, bd, ru, rp = _mixed_inputs(seed, nlev, ncol)
        S = _Mixed(n, nlev, case["levels"], g, bu, bd, case["consistent"], _f0(case))
        nu = ru.numel()
        v = _krylov(S.apply, S.precond, torch.cat([ru, rp]))
        if kind == "mixed":
            return {"u": v[:nu], "p": v[nu:]}
        w = torch.exp(0.5 * torch.cat([_rand(seed, 8, nu), _rand(seed, 9, rp.numel())]))
        # the Krylov method sees the adjoint system in the weights that balance its rows
        D = torch.cat([S.Wh.view(-1), S.Wv.view(-1), S.V.reshape(-1)])
        y = _krylov(lambda t: S.apply_t(D * t) / D, lambda t: S.precond_t(D * t) / D, w * w * v / D)
        lam = D * y
        return {"u": v[:nu], "p": v[nu:], "du": lam[:nu], "dp": lam[nu:]}
    b = _rand(seed, 2, nlev * ncol)
    lv = _hierarchy(n, nlev, case["levels"], g)
    shape = (nlev, ncol)
    if kind == "apply":
        return _apply(lv[0].m, lv[0].a, b.view(shape)).view(-1)
    if kind == "smooth":
        x = _rand(seed, 7, nlev * ncol).view(shape)
        for _ in range(case["sweeps"]):
            x = lv[0].sweep(b.view(shape), x)
        return x.view(-1)
    if kind == "vcycle":
        return _vcycle(lv, b.view(shape)).view(-1)
    x = _solve_h(lv, b)
    if kind == "solve":
        return x
    dz, _ = _vertical(nlev)
    V = (lv[0].m["area"] * dz[:, None]).view(-1)
    w = torch.exp(0.5 * _rand(seed, 8, nlev * ncol))
    lam = V * _solve_h(lv, w * w * x / V)         # H^T = V H V^-1
    X, Lm, m = x.view(shape), lam.view(shape), lv[0].m
    da = torch.zeros(6, nlev, ncol, device=DEV, dtype=torch.float64)
    for s in range(4):
        da[s] = -Lm * (X - X[:, m["nbr"][s]])
    da[4, :-1] = -Lm[:-1] * (X[:-1] - X[1:])
    da[5, 1:] = -Lm[1:] * (X[1:] - X[:-1])
    return {"x": x, "db": lam, "da": da.view(-1)}

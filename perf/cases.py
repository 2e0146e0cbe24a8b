"""Workloads whose speed is tracked: what users of this package have it do,
through its public entry points, over the sizes, boundary kinds, precisions
and forms that are in use.

``listed()`` gives the cases, ``draw(rng)`` one more of the same ranges,
``prepare(case, seed)`` the contexts and buffers a program holds before the
call, ``run(state)`` one pass (some time steps, an adjoint, a half-cell
point) and ``work(case)`` the bytes and operations a pass cannot do without.
``exact(case, seed)`` repeats a pass in double precision with plain torch
operations on whole fields, from the method's equations (no code of the
package but its input generators).

An FP32 context's results are returned in single precision (its populations,
and its adjoint rounded to it); FP64 contexts' in double.
"""
import copy
import math

import numpy as np
import torch

from paper_2409_02930_gb300 import lbm, mea
from paper_2409_02930_gb300 import workloads as W

KINDS = ("slab", "capillary", "batch", "anode", "react", "halfcell", "adjoint")


def listed():
    return [
        # one point of a polarisation curve on a thin electrode slice: the
        # smallest call (48 nodes), a secant on the potential makes many of them
        dict(name="halfcell_12x2x2_f64", kind="halfcell", nx=12, ny=2, nz=2, fp64=True, updates=2, steps=20),
        # binary counter-diffusion tube (1,024 nodes), stepped to steady state
        # in double precision and its molar fluxes read
        dict(name="capillary_256x4_f64", kind="capillary", nx=256, ny=4, fp64=True, steps=100),
        # small electrode slice: the size of quick studies and tests
        dict(name="slab_64x40_f32", kind="slab", nx=64, ny=40, bc="periodic", energy=True, fp64=False, steps=100),
        # the benchmark lattice, single and double precision
        dict(name="slab_512x512_f32", kind="slab", nx=512, ny=512, bc="periodic", energy=True, fp64=False, steps=20),
        dict(name="slab_512x512_f64", kind="slab", nx=512, ny=512, bc="periodic", energy=True, fp64=True, steps=2),
        # the lattice whose state is far larger than the caches
        dict(name="slab_2048x2048_f32", kind="slab", nx=2048, ny=2048, bc="periodic", energy=True, fp64=False,
             steps=4),
        # closed porous sample, ragged sizes (rows that no bulk copy can start on)
        dict(name="slab_701x523_walls_f32", kind="slab", nx=701, ny=523, bc="bounceback", energy=True, fp64=False,
             steps=10),
        # slab fed from a reservoir on each side (the setting of outlet fluxes)
        dict(name="slab_512x384_inlet_f32", kind="slab", nx=512, ny=384, bc="inlet", energy=True, fp64=False,
             steps=10),
        # gradient of an outlet flux with respect to the porosity field
        dict(name="adjoint_256x256_f32", kind="adjoint", nx=256, ny=256, fp64=False, steps=20, ckpt=10),
        # a sweep of 64 tubes of uneven length and pressure in one context
        dict(name="batch_64_f32", kind="batch", cases=64, nmin=128, nmax=4096, lens=5, fp64=False, steps=50),
        # three-dimensional anode, six species, at full size
        dict(name="anode_256x128x128_f32", kind="anode", nx=256, ny=128, nz=128, fp64=False, steps=3),
        # the same gas with the surface mechanism
        dict(name="react_128x64x64_f32", kind="react", nx=128, ny=64, nz=64, fp64=False, steps=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(KINDS, weights=(8, 2, 3, 3, 2, 1, 3))[0]
    fp64 = rng.random() < 0.35
    if kind == "slab":
        fp64 = rng.random() < 0.25
        top = 600 if fp64 else 2048
        nx, ny = _log(rng, 24, top), _log(rng, 24, top)
        if rng.random() < 0.5:
            nx = max(24, nx // 4 * 4)                    # rows of whole 16-byte units half the time
        bc = rng.choice(("periodic", "periodic", "bounceback", "inlet"))
        energy = bc == "inlet" or rng.random() < 0.8
        steps = max(1, min(120, int((6e5 if fp64 else 1.2e7) / (nx * ny))))
        return dict(kind=kind, nx=nx, ny=ny, bc=bc, energy=energy, fp64=fp64, steps=steps)
    if kind == "capillary":
        return dict(kind=kind, nx=_log(rng, 64, 1024), ny=rng.randint(1, 8), fp64=True, steps=rng.randint(40, 120))
    if kind == "batch":
        return dict(kind=kind, cases=_log(rng, 4, 64), nmin=rng.randint(20, 128), nmax=_log(rng, 256, 4096),
                    lens=rng.randint(0, 999), fp64=fp64, steps=rng.randint(20, 60))
    if kind == "anode":
        top = 48 if fp64 else 128
        return dict(kind=kind, nx=_log(rng, 16, 2 * top), ny=_log(rng, 8, top), nz=_log(rng, 4, top), fp64=fp64,
                    steps=rng.randint(1, 3))
    if kind == "react":
        top = 32 if fp64 else 64
        return dict(kind=kind, nx=_log(rng, 12, 2 * top), ny=_log(rng, 4, top), nz=_log(rng, 4, top), fp64=fp64,
                    steps=rng.randint(1, 2))
    if kind == "halfcell":
        return dict(kind=kind, nx=rng.randint(8, 32), ny=rng.randint(2, 4), nz=rng.randint(2, 4), fp64=True,
                    updates=2, steps=rng.randint(8, 20))
    return dict(kind=kind, nx=_log(rng, 32, 256), ny=_log(rng, 32, 256), fp64=fp64, steps=rng.randint(6, 20),
                ckpt=rng.randint(3, 10))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _fed_slab(nx, ny, s, steps):
    """Slab between two reservoirs; next to each face the gas starts at that
    reservoir's composition (blended over eight nodes)."""
    wl = W.slab(nx=nx, ny=ny, seed_phi=s + 1, seed_X=s + 2, steps=steps, bc_x=W.BC_INLET,
                X_lo=[0.8, 0.1, 0.1], X_hi=[0.1, 0.45, 0.45])
    xs = np.tile(np.arange(nx), ny)
    t = xs / max(nx - 1, 1)
    lin = (1 - t)[None] * wl.X_in_lo[:, None] + t[None] * wl.X_in_hi[:, None]
    w = np.minimum(1.0, np.minimum(xs, nx - 1 - xs) / 8.0)
    wl.X_init = (1 - w)[None] * lin + w[None] * wl.X_init
    return wl


def _move_front(wl, rng):
    """Counter-diffusion tube whose two gases meet at a seeded place."""
    xs = np.tile(np.arange(wl.nx), wl.ny)
    left = xs < int(wl.nx * rng.uniform(0.3, 0.7))
    wl.X_init = np.where(left[None], wl.X_in_lo[:, None], wl.X_in_hi[:, None])
    return wl


def _workloads(case, seed):
    """The case's lattices (one, but for a batch) for this seed."""
    s = 1000 + 10 * int(seed)
    rng = np.random.default_rng(s)
    kind = case["kind"]
    if kind == "slab":
        if case["bc"] == "inlet":
            return [_fed_slab(case["nx"], case["ny"], s, case["steps"])]
        wl = W.slab(nx=case["nx"], ny=case["ny"], seed_phi=s + 1, seed_X=s + 2, energy=case["energy"])
        wl.bc_lo = wl.bc_hi = case["bc"]
        return [wl]
    if kind == "adjoint":
        return [_fed_slab(case["nx"], case["ny"], s, case["steps"])]
    if kind == "capillary":
        return [_move_front(W.capillary(nx=case["nx"], ny=case["ny"]), rng)]
    if kind == "batch":
        wls = W.capillary_batch(n_cases=case["cases"], seed=case["lens"], nmin=case["nmin"], nmax=case["nmax"])
        return [_move_front(w, rng) for w in wls]
    mech = None
    if kind == "react":
        mech = W.surface_mechanism()
    if kind == "halfcell":
        mech = W.surface_mechanism(electrochem=True)
    return [W.anode3d(nx=case["nx"], ny=case["ny"], nz=case["nz"], seed_phi=s + 1, seed_X=s + 2, mechanism=mech)]


def _potential(seed):
    return 0.2 + 0.3 * float(np.random.default_rng(77 + int(seed)).random())


def prepare(case, seed):
    wls = _workloads(case, seed)
    prec = lbm.LBM_FP64 if case["fp64"] else lbm.LBM_FP32
    dt = torch.float64 if case["fp64"] else torch.float32
    s = {"case": case, "wls": wls}
    g = s["g"] = lbm.Batch(wls, precision=prec) if case["kind"] == "batch" else lbm.Lattice(wls[0], precision=prec)
    if case["kind"] == "adjoint":
        return s
    s["pops"] = torch.empty(g.L * g.Q * g.N, dtype=dt, device="cuda")
    if case["kind"] in ("react", "halfcell"):
        s["xs"] = torch.empty((wls[0].mechanism.S, g.N), dtype=torch.float64, device="cuda")
    if case["kind"] == "capillary" and case["fp64"]:
        s["flux"] = torch.empty((g.M, g.D, g.N), dtype=torch.float64, device="cuda")
    if case["kind"] == "halfcell":
        wl = wls[0]
        s["image"] = g.save()
        s["cell"] = mea.HalfCell(g, wl.nx, wl.ny, wl.nz, wl.dx, wl.mechanism.resistivity)
        s["potential"] = _potential(seed)
    return s


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

def _populations(s):
    g, buf = s["g"], s["pops"]
    lib = lbm.load()
    g._check(lib.lbm_get_populations(g._h, buf.data_ptr(), buf.numel() * buf.element_size(), 1), "populations")
    if s["case"]["kind"] == "batch":
        return [buf]                                     # case after case, as the library lays them out
    return list(buf.view(g.L, g.Q, g.N))


def run(s):
    case, g = s["case"], s["g"]
    kind = case["kind"]
    if kind == "adjoint":
        J, dphi, dpore, dtort = g.adjoint(case["steps"], case["ckpt"])
        real = np.float64 if case["fp64"] else np.float32
        return {"J": np.array([J], real), "dphi": dphi.astype(real), "dpore": np.array([dpore], real),
                "dtort": np.array([dtort], real)}
    out = {}
    if kind == "halfcell":
        st = s["cell"].polarisation_curve([s["potential"]], restore=lambda: g.load_state(s["image"]),
                                          steps_per_update=case["steps"], max_updates=case["updates"], tol=0.0)[0]
        out.update(Iv=st.Iv_x, Ia=st.Ia_x, phi_el=st.phi_electrolyte)
    else:
        g.step(case["steps"])
    out["pops"] = _populations(s)
    if "flux" in s:
        out["flux"] = g.moments_device(lbm.LBM_MOM_N_A, s["flux"])
    if "xs" in s:
        out["xs"] = g.moments_device(lbm.LBM_MOM_XS, s["xs"])
    return out


def work(case):
    """Every time step reads and writes each population once and reads the
    porosity (and coverages) once; operations are those of the relaxation
    written out per population, and of the surface solve per step."""
    kind, rb = case["kind"], 8 if case["fp64"] else 4
    d3 = kind in ("anode", "react", "halfcell")
    M = 6 if d3 else (2 if kind in ("capillary", "batch") else 3)
    L = M + 1 + (0 if kind in ("capillary", "batch") or not case.get("energy", True) else 1)
    Q = 27 if d3 else 9
    if kind == "batch":
        N = sum(w.N for w in W.capillary_batch(n_cases=case["cases"], seed=case["lens"], nmin=case["nmin"],
                                               nmax=case["nmax"]))
    else:
        N = case["nx"] * case["ny"] * case.get("nz", 1)
    node_b = 2 * L * Q * rb + rb
    node_f = L * Q * (10 + 2 * M) + 150
    if kind in ("react", "halfcell"):
        node_b += 2 * 8 * 8
        node_f += 6000
    steps = case["steps"] * case.get("updates", 1)
    if kind == "adjoint":
        # forward, recomputation of all but one step of each segment, reverse
        # sweep (state, adjoint in, adjoint out) at about three evaluations
        node_b, node_f = 3 * node_b, 5 * node_f
    return {"bytes": float(N) * node_b * steps, "flops": float(N) * node_f * steps}


# --------------------------------------------------------------------------
# the same pass in double precision
# --------------------------------------------------------------------------

RU_SI, FARADAY = 8.314462618, 96485.33212


def _dev(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device="cuda")


class _Exact:
    """Whole-field double-precision form of one lattice's step; fields are
    [..., nz, ny, nx] (nz = 1 in two dimensions)."""

    def __init__(self, wl, phi=None, lam=None):
        self.w, self.M, self.D = wl, wl.M, wl.D
        self.shape = (wl.nz, wl.ny, wl.nx)
        zs = (-1, 0, 1) if wl.D == 3 else (0,)
        self.c = [(x, y, z) for z in zs for y in (-1, 0, 1) for x in (-1, 0, 1)]
        self.Q, self.L = len(self.c), wl.L
        m = np.asarray(wl.molar_mass)
        self.dt = wl.dx * math.sqrt(wl.theta_max * m.min() / (RU_SI * wl.T_scale))
        self.cv = wl.dx / self.dt
        c2 = self.cv ** 2
        self.RU = RU_SI / c2
        self.m, self.Ra = m, self.RU / m
        self.cvR = np.asarray(wl.cv_factor) * self.Ra
        self.U0 = np.asarray(wl.U0) / c2
        self.phi = phi if phi is not None else _dev(wl.porosity).view(self.shape)
        self.lam = 1.0 if lam is None else lam
        self.T0 = _dev(wl.T_init).view(self.shape)
        if wl.mechanism is not None:
            self.Xs = _dev(wl.mechanism.Xs_init).view(-1, 1, 1, 1).expand(-1, *self.shape).clone()
            self.dphi = torch.full(self.shape, float(wl.mechanism.dphi), dtype=torch.float64, device="cuda")
        X, P = _dev(wl.X_init).view(-1, *self.shape), _dev(wl.P_init).view(self.shape)
        rho_a = [P * X[a] * m[a] / (RU_SI * self.T0) for a in range(self.M)]
        u = [torch.zeros_like(P) for _ in range(self.D)]
        self.f = self.equilibrium(self.phi, rho_a, u, self.T0)

    def form(self, xi, P):
        """Product form [Q, ...] of per-axis parameters xi, P."""
        ax = [torch.stack([(p - x) / 2, 1 - p, (p + x) / 2]) for x, p in zip(xi, P)]
        v = ax[1][:, None] * ax[0][None]
        if self.D == 3:
            v = ax[2][:, None, None] * v[None]
        return v.reshape(self.Q, *v.shape[self.D:])

    def geq(self, phi, rho, u, RT, U):
        w = [a / phi for a in u]
        one = [(x, RT + x * x) for x in w]
        two = [(RT * x + x ** 3 / 2, RT ** 2 + 2.5 * RT * x * x + x ** 4 / 2, x * x / 2) for x in w]
        f1 = [torch.stack([(p - x) / 2, 1 - p, (p + x) / 2]) for x, p in one]
        f2 = [torch.stack([(p - x) / 2, z - p, (p + x) / 2]) for x, p, z in two]

        def prod(fs):
            v = fs[1][:, None] * fs[0][None]
            if self.D == 3:
                v = fs[2][:, None, None] * v[None]
            return v.reshape(self.Q, *v.shape[self.D:])
        s = U * prod(f1)
        for b in range(self.D):
            s = s + prod([f2[a] if a == b else f1[a] for a in range(self.D)])
        return phi * rho * s

    def equilibrium(self, phi, rho_a, u, T):
        rho = sum(rho_a)
        Rg = self.RU * sum(r / rho / m for r, m in zip(rho_a, self.m))
        w = [a / phi for a in u]
        pops = [phi * r * self.form(w, [x * x + Ra * T for x in w]) for r, Ra in zip(rho_a, self.Ra)]
        pops.append(phi * rho * self.form(w, [x * x + Rg * T for x in w]))
        if self.w.energy:
            U = sum(r / rho * (u0 + c * (T - self.w.T_thermo)) for r, u0, c in zip(rho_a, self.U0, self.cvR))
            pops.append(self.geq(phi, rho, u, Rg * T, U))
        return torch.stack(pops)

    def stream(self):
        f, w, out = self.f, self.w, []
        for i, (cx, cy, cz) in enumerate(self.c):
            out.append(torch.roll(f[:, i], (cz, cy, cx), (1, 2, 3)))
        for side, bc in ((0, w.bc_lo), (1, w.bc_hi)):
            if bc == W.BC_PERIODIC:
                continue
            xb, xa, into = (0, 1, 1) if side == 0 else (w.nx - 1, w.nx - 2, -1)
            if bc == W.BC_BOUNCEBACK:
                new = [f[:, self.Q - 1 - i, :, :, xb] for i in range(self.Q)]
            else:
                a = torch.stack([o[self.M, :, :, xa] for o in out])
                rho_f = a.sum(0) / self.phi[:, :, xa]
                u = [sum(c[b] * a[i] for i, c in enumerate(self.c)) / rho_f for b in range(self.D)]
                T, P, X = ((w.T_in_lo, w.P_in_lo, w.X_in_lo), (w.T_in_hi, w.P_in_hi, w.X_in_hi))[side]
                pb = self.phi[:, :, xb]
                new = self.equilibrium(pb, [P * x * m / (RU_SI * T) * torch.ones_like(pb) for x, m in zip(X, self.m)],
                                       u, T * torch.ones_like(pb))
                new = [new[:, i] for i in range(self.Q)]
            for i, c in enumerate(self.c):
                if c[0] == into:
                    o = out[i]
                    parts = [new[i][..., None], o[..., 1:]] if side == 0 else [o[..., :-1], new[i][..., None]]
                    out[i] = torch.cat(parts, -1)
        return torch.stack(out, 1)

    def shift(self, a, axis, by):
        """Neighbour values at +by along axis (0: x), edge copy at open x faces."""
        if axis > 0 or self.w.bc_lo == W.BC_PERIODIC:
            return torch.roll(a, -by, -1 - axis)
        return torch.cat([a[..., 1:], a[..., -1:]], -1) if by > 0 else torch.cat([a[..., :1], a[..., :-1]], -1)

    def grad(self, a, axis):
        for b in range(self.D):
            if b != axis:
                a = a * (2 / 3) + (self.shift(a, b, 1) + self.shift(a, b, -1)) / 6
        return (self.shift(a, axis, 1) - self.shift(a, axis, -1)) / 2

    def macro(self, f):
        w, M, D, phi = self.w, self.M, self.D, self.phi
        mom = lambda l, b: sum(c[b] * f[l, i] for i, c in enumerate(self.c) if c[b])  # noqa: E731
        s = {"rho_a": [f[a].sum(0) / phi for a in range(M)], "rho": f[M].sum(0) / phi}
        s["ja"] = [[mom(a, b) for b in range(D)] for a in range(M)]
        s["u"] = [mom(M, b) / s["rho"] for b in range(D)]
        rho_s = sum(s["rho_a"])
        s["rho_s"] = rho_s
        s["Y"] = [r / rho_s for r in s["rho_a"]]
        inv_m = sum(y / m for y, m in zip(s["Y"], self.m))
        s["mm"], s["R"] = 1 / inv_m, self.RU * inv_m
        s["cv"] = sum(y * c for y, c in zip(s["Y"], self.cvR))
        s["w"] = [a / phi for a in s["u"]]
        w2 = sum(x * x for x in s["w"])
        if w.energy:
            E = f[M + 1].sum(0) / (phi * s["rho"])
            s["T"] = w.T_thermo + (E - w2 / 2 - sum(y * u for y, u in zip(s["Y"], self.U0))) / s["cv"]
            s["q"] = [mom(M + 1, b) for b in range(D)]
        else:
            s["T"] = self.T0
        s["P"] = s["rho"] * s["R"] * s["T"]
        s["Pi"] = [s["rho"] * u * (1 - 3 * s["R"] * s["T"]) - s["rho"] * u * x * x for u, x in zip(s["u"], s["w"])]
        return s

    def transport(self, s):
        w, M, D = self.w, self.M, self.D
        T = s["T"]
        D_si = np.asarray(w.D_ref) / (self.cv * w.dx)
        tr = T / w.T_ref
        C = s["mm"] * self.RU * T * s["P"] / (w.P_ref / self.cv ** 2 * tr ** 1.5)
        kap = [[C / (D_si[a, b] * self.m[a] * self.m[b]) if a != b else None for b in range(M)] for a in range(M)]
        it = [sum(s["Y"][b] * kap[a][b] for b in range(M) if b != a) for a in range(M)]
        itk = [torch.zeros_like(T)] * M
        if w.knudsen:
            d0 = 2 * w.pore_radius / w.dx
            itk = [self.lam * 3 * w.tortuosity * self.RU * T / (d0 * self.phi * m * torch.sqrt(8 * self.RU * T / (math.pi * m)))
                   for m in self.m]
        A = [[1 + it[a] / 2 + itk[a] / 2 if a == b else -s["Y"][b] * kap[a][b] / 2 for b in range(M)] for a in range(M)]
        B = []
        for a in range(M):
            tiny = s["rho_a"][a] < 1e-14 * s["rho_s"]
            safe = torch.where(tiny, torch.ones_like(tiny, dtype=torch.float64), s["rho_a"][a])
            B.append([torch.where(tiny, torch.zeros_like(T), s["ja"][a][b] / safe - s["u"][b])
                      - itk[a] / 2 * s["u"][b] for b in range(D)])
        for k in range(M):                                # the matrix is diagonally dominant
            for r in range(k + 1, M):
                f = A[r][k] / A[k][k]
                A[r] = [A[r][c] - f * A[k][c] if c > k else A[r][c] for c in range(M)]
                B[r] = [B[r][b] - f * B[k][b] for b in range(D)]
        V = [None] * M
        for k in reversed(range(M)):
            V[k] = [(B[k][b] - sum(A[k][j] * V[j][b] for j in range(k + 1, M))) / A[k][k] for b in range(D)]
        return kap, [i / (2 + i) for i in it], itk, V

    def surface(self, s):
        """Backward-Euler extents of the surface steps; species production,
        new coverages, internal-energy change and volumetric current."""
        w, M, mc = self.w, self.M, self.w.mechanism
        R, S = mc.R, mc.S
        edge = np.zeros(R) if mc.edge is None else np.asarray(mc.edge, float)
        nel = np.zeros(R) if mc.edge is None else np.asarray(mc.n_el, float)
        T, phi, dphi = s["T"].reshape(-1), self.phi.reshape(-1), self.dphi.reshape(-1)
        nu = _dev(np.concatenate([mc.nu_gas, mc.nu_surf], 1))                     # [R, S + M]
        es = _dev(np.where(edge > 0, mc.l_tpb / mc.a_s, 1.0))
        kr = _dev(mc.A)[:, None] * torch.exp(-_dev(mc.Ea)[:, None] / (RU_SI * T))
        kr = kr * es[:, None] * torch.exp(_dev(edge * nel * mc.beta_ct)[:, None] * FARADAY * dphi / (RU_SI * T))
        N = T.numel()
        scale = torch.cat([(mc.a_s / phi).expand(M, N), torch.ones(S, N, dtype=T.dtype, device=T.device)])
        c0 = torch.cat([torch.stack([r.reshape(-1) / m for r, m in zip(s["rho_a"], self.m)]),
                        mc.gamma * self.Xs.reshape(S, N)])
        order = (-nu).clamp(min=0).cpu().numpy()
        xi, done = torch.zeros(R, N, dtype=T.dtype, device=T.device), torch.zeros(N, dtype=torch.bool, device=T.device)
        best = torch.full((N,), math.inf, dtype=T.dtype, device=T.device)
        eye = torch.eye(R, dtype=T.dtype, device=T.device)
        for _ in range(40):
            c = c0 + scale * (nu.T @ xi)
            pos, r = c.clamp(min=0), []
            for k in range(R):
                v = kr[k]
                for j in np.nonzero(order[k])[0]:
                    v = v * pos[j] ** int(order[k][j])
                r.append(v)
            r = torch.stack(r)
            U = self.dt * r[:, None] * _dev(order)[..., None] * torch.where(c > 0, 1 / c, 0.0)[None]   # [R, NS, N]
            J = eye - torch.einsum("kin,in,li->nkl", U, scale, nu)
            d = torch.linalg.solve(J, -(xi - self.dt * r).T[..., None])[..., 0].T
            dc = scale * (nu.T @ d)
            lim = torch.where((c >= 0) & (c + dc < 0), 0.9 * c / (-dc), torch.ones_like(c)).amin(0)
            step = torch.where(done, torch.zeros_like(lim), lim)
            xi = xi + step * d
            size = (step * d).abs().amax(0) / (xi.abs().amax(0) + 1e-300)
            done = done | ((lim == 1) & ((size <= 1e-14) | ((size <= 1e-12) & (size >= best))))
            best = torch.minimum(best, size)
            if bool(done.all()):
                break
        dn = nu.T @ xi
        rd = [(mc.a_s * m * dn[a]).view(self.shape) for a, m in enumerate(self.m)]
        Xs = self.Xs + (dn[M:] / mc.gamma).view(S, *self.shape)
        Us = _dev(mc.surf_U0)[:, None] + _dev(mc.surf_cv_factor)[:, None] * RU_SI * (T - w.T_thermo)
        cur = FARADAY * mc.a_s * (_dev(edge * nel)[:, None] * xi).sum(0) / self.dt
        src = 0.0
        if mc.l_tpb > 0:
            src = (mc.a_s / mc.l_tpb * cur ** 2 * mc.resistivity * w.dx - dphi.abs() * cur) * self.dt
        dU = ((src - mc.a_s * (dn[M:] * Us).sum(0)) / self.cv ** 2).view(self.shape)
        return rd, Xs, dU, cur.view(self.shape)

    def current(self):
        return self.surface(self.macro(self.stream()))[3].reshape(-1).cpu().numpy()

    def step(self):
        w, M, D, phi = self.w, self.M, self.D, self.phi
        f = self.stream()
        s = self.macro(f)
        kap, beta, itk, V = self.transport(s)
        u, x, T, rho, Y = s["u"], s["w"], s["T"], s["rho"], s["Y"]
        divu = sum(self.grad(u[b], b) for b in range(D))
        dPi = [self.grad(s["Pi"][b], b) for b in range(D)]
        rd = None
        if w.mechanism is not None:
            rd, self.Xs, dU, _ = self.surface(s)
        E, S, K = [], [], []
        zero = torch.zeros_like(T)
        for a in range(M):
            t, pr = self.Ra[a] * T, phi * s["rho_a"][a]
            xs = [(u[b] + V[a][b]) / phi for b in range(D)]
            E.append(pr * self.form(x, [v * v + t for v in x]))
            S.append(pr * self.form(xs, [v * v + t for v in xs]))
            K.append(pr * self.form([zero] * D, [t] * D))
        new = []
        for a in range(M):
            F = Y[a] * sum(kap[a][b] * (E[b] - S[b]) for b in range(M) if b != a) + itk[a] * (S[a] - K[a])
            o = f[a] + 2 * beta[a] * (E[a] - f[a]) + (beta[a] - 1) * F
            if rd is not None:
                o = o + rd[a] * self.form(x, [v * v + self.Ra[a] * T for v in x])
            new.append(o)
        del E, S, K
        mu = sum(s["mm"] * y / m * r for y, m, r in zip(Y, self.m, np.asarray(w.mu_ref) / (self.cv * w.dx)))
        mu = mu * (T / w.T_ref) ** w.mu_exp
        om, om1 = 1 / (0.5 + mu / s["P"]), 1 / (0.5 + mu / (w.Pr * s["P"]))
        bulk = -w.bulk_ratio * mu + mu * (2 / D - (s["R"] / s["cv"] if w.energy else 0.0))
        drag = 1 + 0.5 * sum(r * k for r, k in zip(s["rho_a"], itk)) / rho
        Vbar = [sum(Y[a] * V[a][b] for a in range(M)) for b in range(D)]
        xe, Pe = [], []
        for b in range(D):
            Fk = -sum(s["rho_a"][a] * (u[b] + V[a][b] - Vbar[b]) * itk[a] for a in range(M)) / drag
            xe.append((u[b] + Fk / (om * rho)) / phi)
            Pe.append(s["R"] * T + x[b] * x[b] + bulk * divu / (phi * rho) + (2 - om) / (2 * om * phi * rho) * dPi[b])
        fex = phi * rho * self.form(xe, Pe)
        o = f[M] + om * (fex - f[M])
        rho_pc = rho
        if rd is not None:
            rho_pc = rho + sum(rd) / phi
            o = o + (rho_pc / rho - 1) * fex
        new.append(o)
        if w.energy:
            Ua = [self.U0[a] + self.cvR[a] * (T - w.T_thermo) for a in range(M)]
            Ha = [Ua[a] + self.Ra[a] * T for a in range(M)]
            U, RT = sum(y * v for y, v in zip(Y, Ua)), s["R"] * T
            w2 = sum(v * v for v in x)
            g = f[M + 1]
            geq = self.geq(phi, rho, u, RT, U)
            o = g + om * (geq - g)
            if rd is not None:
                o = o + self.geq(phi, rho_pc, u, RT, (phi * rho * U + dU) / (phi * rho_pc)) - geq
            o = list(o)
            for b in range(D):
                uP = zero
                for c in range(D):
                    Pt = sum(d[b] * d[c] * f[M, i] for i, d in enumerate(self.c) if d[b] * d[c])
                    uP = uP + x[c] * (Pt - rho * u[b] * x[c] - (phi * rho * RT if b == c else 0.0))
                sV = sum(Ha[a] * Y[a] * (V[a][b] - Vbar[b]) for a in range(M))
                sdY = sum(Ha[a] * self.grad(Y[a], b) for a in range(M))
                Dq = (om - om1) * (s["q"][b] - uP - (U + RT + w2 / 2) * rho * u[b]) + om1 * rho * sV \
                    + 0.5 * (2 - om1) * s["P"] * phi * sdY + u[b] * om * bulk * divu / phi \
                    - 0.5 * (om - om1) * x[b] * dPi[b]
                for i, c in enumerate(self.c):
                    if sum(v * v for v in c) == 1 and c[b]:
                        o[i] = o[i] + 0.5 * c[b] * Dq
            new.append(torch.stack(o))
        self.f = torch.stack(new)


def _steps(wl, n):
    e = _Exact(wl)
    for _ in range(n):
        e.step()
    return e


def _exact_adjoint(case, wl):
    phi = _dev(wl.porosity).view(1, wl.ny, wl.nx).requires_grad_(True)
    lam = torch.ones((), dtype=torch.float64, device="cuda", requires_grad=True)
    e = _Exact(copy.copy(wl), phi, lam)
    for _ in range(case["steps"]):
        e.step()
    J = e.macro(e.stream())["ja"][0][0][:, :, wl.nx - 2].sum()
    J.backward()
    dl = float(lam.grad)
    one = lambda v: np.array([float(v)])  # noqa: E731
    return {"J": one(J.detach()), "dphi": phi.grad.reshape(-1).cpu().numpy(), "dpore": one(-dl / wl.pore_radius),
            "dtort": one(dl / wl.tortuosity)}


def exact(case, seed):
    wls, kind = _workloads(case, seed), case["kind"]
    flat = lambda e: e.f.reshape(e.L, e.Q, -1)  # noqa: E731
    if kind == "adjoint":
        return _exact_adjoint(case, wls[0])
    with torch.no_grad():
        if kind == "batch":
            return {"pops": [torch.cat([flat(_steps(w, case["steps"])).reshape(-1) for w in wls])]}
        if kind == "halfcell":
            wl, e = wls[0], _Exact(wls[0])
            om, el = wl.mechanism.resistivity, np.zeros(wl.nx)
            for _ in range(case["updates"]):
                e.dphi = _dev(np.broadcast_to(_potential(seed) - el, e.shape).copy())
                for _ in range(case["steps"]):
                    e.step()
                Iv = e.current().reshape(e.shape).mean(axis=(0, 1))
                Ia = np.cumsum(Iv) * wl.dx
                el = np.concatenate([[0.0], np.cumsum((Ia * om * wl.dx)[:-1])])
            return {"Iv": Iv, "Ia": Ia, "phi_el": el, "pops": list(flat(e)), "xs": e.Xs.reshape(len(e.Xs), -1)}
        e = _steps(wls[0], case["steps"])
        out = {"pops": list(flat(e))}
        if kind == "react":
            out["xs"] = e.Xs.reshape(len(e.Xs), -1)
        if kind == "capillary" and case["fp64"]:
            s = e.macro(e.stream())
            V = e.transport(s)[3]
            out["flux"] = torch.stack([torch.stack([s["rho_a"][a] * (s["u"][b] + V[a][b]) * e.cv / e.m[a]
                                                    for b in range(e.D)]) for a in range(e.M)]).reshape(e.M, e.D, -1)
        return out

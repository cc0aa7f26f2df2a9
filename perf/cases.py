"""Workloads that a user of this library runs, each one pass through its public entry points.

A case is a dict of plain values: the kind of call, the mesh (nx, ny, nz elements of mean width h bohr,
uniform or graded 1.25 toward the nuclei, degree p), the orbitals, the nuclei and the arithmetic.

Arithmetic: FP64 (the default of every call), double-float and the relaxed schedule.  FP32 alone and BF16
operands miss the bound on the dipole error and are there for accuracy studies, so no case uses them by
themselves; the relaxed schedule runs FP32 products inside each exponential.

`exact` computes what a case returns in 64 bits with plain torch: quadrature tables, the element operator
with one index array per axis, Chebyshev exponentials, a dense fast-diagonalization Poisson solve, the
LDA formula and, for the objective, torch autograd through all of it.
"""
import math

import numpy as np
import torch

from paper_1810_13130_gb300 import tdks

PREC = {"fp64": tdks.FP64, "df64": tdks.DF64, "mixed": tdks.MIXED}
KICK = 1e-3
C128, F64 = torch.complex128, torch.float64


def listed():
    mol = dict(h=2.0, p=6, grid="uniform", nuc="erf")
    atom = dict(nx=6, ny=6, nz=6, h=10.0 / 3.0, p=4, n_orb=1, n_nuc=1, grid="uniform", nuc="soft")
    return [
        # Hbar psi of the two-electron atom (the smallest workload): launch latency.
        dict(name="apply_atom", kind="apply", prec="fp64", **atom),
        # An odd, graded mesh of odd degree with few orbitals: padding and ragged tiles.
        dict(name="apply_ragged", kind="apply", nx=11, ny=7, nz=9, h=1.5, p=5, n_orb=3, n_nuc=2, grid="graded",
             nuc="soft", prec="fp64"),
        # The molecule's Hbar psi, as an eigensolver or an own propagator calls it.
        dict(name="apply_molecule", kind="apply", nx=16, ny=16, nz=16, n_orb=16, n_nuc=8, prec="fp64", **mol),
        # All-electron-like: bare nuclei on a graded mesh at the highest degree, double-float.
        dict(name="apply_graded_df64", kind="apply", nx=20, ny=20, nz=20, h=1.6, p=8, n_orb=5, n_nuc=5,
             grid="graded", nuc="bare", prec="df64"),
        # One exponential with nonlocal projectors on every atom (a user's own time stepping).
        dict(name="expm_projectors", kind="expm", nx=8, ny=8, nz=8, n_orb=8, n_nuc=4, dt=0.1, kb=True, prec="fp64",
             **mol),
        # The same call on a long thin molecule in the relaxed schedule.
        dict(name="expm_relaxed", kind="expm", nx=18, ny=10, nz=8, n_orb=12, n_nuc=6, dt=0.1, kb=False, prec="mixed",
             **mol),
        # Density, Hartree, LDA and dipole of two successive orbital sets (the field part of a step,
        # the second Poisson solve warm-started by the first).
        dict(name="fields_molecule", kind="fields", nx=14, ny=14, nz=14, n_orb=10, n_nuc=6, **mol),
        # The atom's propagation: many small launches.
        dict(name="steps_atom", kind="steps", dt=0.05, steps=4, prec="fp64", **atom),
        # One step of the benchmarked molecule (16^3 elements, 16 orbitals) in the default arithmetic.
        dict(name="steps_molecule", kind="steps", nx=16, ny=16, nz=16, n_orb=16, n_nuc=8, dt=0.1, steps=1,
             prec="fp64", **mol),
        # A mid-size molecule in double-float.
        dict(name="steps_molecule_df64", kind="steps", nx=8, ny=8, nz=8, n_orb=8, n_nuc=4, dt=0.1, steps=2,
             prec="df64", **mol),
        # Many uneven systems per step (degrees 4..8, 1..8 orbitals) in the relaxed schedule.
        dict(name="batch_relaxed", kind="batch", n_sys=12, n_lo=4, n_hi=9, seed=5, steps=1, prec="mixed"),
        # The objective of pulse shaping and its gradient with respect to the field.
        dict(name="gradient_atom", kind="gradient", dt=0.1, steps=8, ckpt=4, prec="fp64", **atom),
    ]


def draw(rng):
    """A further case of the same kinds and ranges, no dearer than the dearest listed one."""
    kind = rng.choice(["apply", "apply", "expm", "fields", "steps", "batch", "gradient"])
    if kind == "batch":
        return dict(kind=kind, n_sys=rng.randint(3, 12), n_lo=rng.randint(2, 5), n_hi=rng.randint(5, 9),
                    seed=rng.randint(10, 10 ** 6), steps=rng.randint(1, 2), prec=rng.choice(["fp64", "df64", "mixed"]))
    limit = 6e9 if kind == "gradient" else 2e12          # flops: a pass within the listed cases' range
    while True:
        p = rng.choice([2, 3, 4, 4, 5, 5, 6, 6, 7, 8])
        c = dict(kind=kind, p=p, h=round(rng.uniform(0.3, 0.5) * p, 3), grid=rng.choice(["uniform", "graded"]),
                 nuc=rng.choice(["soft", "erf"]))
        for d in ("nx", "ny", "nz"):
            c[d] = int(round(2 ** rng.uniform(1, 4.3)))
        c["n_orb"] = int(round(2 ** rng.uniform(0, 4)))
        c["n_nuc"] = rng.randint(1, max(1, c["n_orb"] // 2))
        if kind != "fields":
            c["prec"] = "fp64" if kind == "gradient" else rng.choice(["fp64", "fp64", "df64", "mixed"])
        if kind in ("expm", "steps", "gradient"):
            c["dt"] = rng.choice([0.02, 0.05, 0.1])
        if kind == "expm":
            c["kb"] = rng.random() < 0.3
        if kind == "steps":
            c["steps"] = rng.randint(1, 3)
        if kind == "gradient":
            c["n_orb"] = min(c["n_orb"], 3)
            c.update(steps=rng.randint(3, 8), ckpt=rng.randint(2, 4))
            if c["dt"] * _half_width(c) > 15.0:          # the adjoint takes no sub-steps
                continue
        if work(c)["flops"] <= limit and 300 * c["n_orb"] ** 2 <= _n_int(c) * c["n_orb"] <= 14e6:
            return c


# ---- what a program has in hand before the call ------------------------------------------------------------

def _breaks(n, h, grid):
    if grid == "uniform":
        return np.linspace(-0.5 * n * h, 0.5 * n * h, n + 1)
    w = 1.25 ** np.abs(np.arange(n) - 0.5 * (n - 1))
    e = np.concatenate([[0.0], np.cumsum(w)]) / w.sum()
    return (e - 0.5) * n * h


def _n_int(c):
    return (c["nx"] * c["p"] - 1) * (c["ny"] * c["p"] - 1) * (c["nz"] * c["p"] - 1)


def _system(c, rng):
    """Mesh and nuclei: breakpoints, positions in the middle of the box, charges."""
    br = [_breaks(c[d], c["h"], c["grid"]) for d in ("nx", "ny", "nz")]
    half = np.array([b[-1] for b in br])
    if c["n_nuc"] == 1 and c["nuc"] == "soft":
        R = rng.uniform(-0.05, 0.05, (1, 3))
    else:
        R = rng.uniform(-1.0, 1.0, (c["n_nuc"], 3)) * np.minimum(half / 3.0, 6.0)
    Z = {"soft": 2.0, "erf": 4.0, "bare": 6.0}[c["nuc"]] * np.ones(c["n_nuc"])
    return dict(br=br, R=R, Z=Z, p=c["p"], n_orb=c["n_orb"], nuc=c["nuc"],
                par={"soft": 0.5, "erf": 0.8, "bare": 0.0}[c["nuc"]])


def _orbitals(c, seed):
    """Orthonormal smooth orbitals [n_orb, n_int]: Gaussians times linear polynomials and a phase in the
    normalized node index, x fastest."""
    rng = np.random.default_rng([seed, 77])
    dev = torch.device("cuda")
    ax = [torch.arange(1, c[d] * c["p"], device=dev, dtype=F64) / (c[d] * c["p"]) for d in ("nx", "ny", "nz")]
    cols = []
    for _ in range(c["n_orb"]):
        cen, w = rng.uniform(0.4, 0.6, 3), rng.uniform(0.07, 0.12)
        g = [torch.exp(-(ax[d] - cen[d]) ** 2 / (2 * w * w)) for d in range(3)]
        lin = [rng.uniform(-3, 3) * (ax[d] - cen[d]) for d in range(3)]
        poly = 1.0 + lin[2][:, None, None] + lin[1][None, :, None] + lin[0][None, None, :]
        ph = torch.exp(1j * rng.uniform(-2, 2) * (ax[0] - cen[0]))
        cols.append((poly * g[2][:, None, None] * g[1][None, :, None] * (g[0] * ph)[None, None, :]).reshape(-1))
    A = torch.stack(cols)
    for _ in range(2):
        L = torch.linalg.cholesky((A @ A.conj().T).cpu())
        A = torch.linalg.inv(L).to(dev) @ A
    return A.contiguous()


def _context(c, s):
    ctx = tdks.Context(*s["br"], s["p"], s["n_orb"], np.full(s["n_orb"], 2.0), s["R"], s["Z"], s["nuc"], s["par"])
    ctx.set_cg(1e-12)
    return ctx


def _potential(c, s, seed):
    """A self-consistent-looking V_KS: the nuclear potential plus a smooth repulsive part and some noise."""
    ref = _Ref(s)
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = ref.v_nuc()
    return (v * 0.7 + 0.05 * torch.rand(v.shape, generator=g, device="cuda", dtype=F64)).contiguous()


def _fields_E(c, seed):
    rng = np.random.default_rng([seed, 3])
    return rng.uniform(-5e-3, 5e-3, (c["steps"], 6))


def _batch_cases(c):
    """Uneven systems: n^3 elements, degrees 4..8, 1..8 orbitals, their own time steps."""
    rng = np.random.default_rng(c["seed"])
    out = []
    for _ in range(c["n_sys"]):
        n = [int(rng.integers(c["n_lo"], c["n_hi"] + 1)) for _ in range(3)]
        out.append(dict(nx=n[0], ny=n[1], nz=n[2], h=2.0, p=int(rng.integers(4, 9)), n_orb=int(rng.integers(1, 9)),
                        n_nuc=int(rng.integers(2, 5)), grid="uniform", nuc="soft", prec=c["prec"],
                        dt=float(rng.choice([0.02, 0.05, 0.1]))))
    return out


class _Cfg:
    """A system as tdks.Batch takes it."""

    def __init__(self, s):
        self.X, self.Y, self.Z = s["br"]
        self.p, self.nq, self.n_orb, self.occ = s["p"], 0, s["n_orb"], np.full(s["n_orb"], 2.0)
        self.atom_R, self.atom_Z, self.nuc_kind, self.nuc_param = s["R"], s["Z"], s["nuc"], s["par"]
        self.hartree = self.xc = True


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "batch":
        subs = _batch_cases(c)
        ss = [_system(q, np.random.default_rng([seed, k])) for k, q in enumerate(subs)]
        b = tdks.Batch([_Cfg(s) for s in ss], [q["dt"] for q in subs], prec=PREC[c["prec"]])
        return dict(case=c, b=b, psi=[_orbitals(q, seed + 1000 * k) for k, q in enumerate(subs)])
    s = _system(c, np.random.default_rng([seed, 0]))
    ctx = _context(c, s)
    st = dict(case=c, ctx=ctx, psi=_orbitals(c, seed))
    if kind in ("apply", "expm"):
        ctx.set_potential(_potential(c, s, seed))
    if kind == "expm" and c["kb"]:
        ctx.set_kb(s["R"])
    if kind == "fields":
        st["psi2"] = _orbitals(c, seed + 500)
    if kind == "steps":
        ctx.kick(st["psi"], KICK, (1.0, 0.0, 0.0))
        st.update(work=torch.empty_like(st["psi"]), E=_fields_E(c, seed))
    if kind == "gradient":
        st["E"] = torch.from_numpy(_fields_E(c, seed)).requires_grad_(True)
    return st


def _half_width(c):
    """Spectral half-width of Hbar: the largest eigenvalue of -d^2/dx^2 on GLL elements of degree p and width h
    is (0.48 + 3.8 / p^2) p^4 / h^2 within 3 % for p = 2..8."""
    h = [np.diff(_breaks(c[d], c["h"], c["grid"])).min() for d in ("nx", "ny", "nz")]
    return sum(0.25 * (0.48 + 3.8 / c["p"] ** 2) * c["p"] ** 4 / x ** 2 for x in h)


def _weights(c):
    w = np.full(c["steps"] + 1, c["dt"])
    w[0] = w[-1] = 0.5 * c["dt"]
    return w


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "batch":
        b = state["b"]
        for k, p in enumerate(state["psi"]):
            b.set_orbitals(k, p)
        d0 = b.init()
        d = b.steps(c["steps"])
        return {"d0": d0, "d": d, "psi": [b.get_orbitals(k) for k in range(b.n_sys)]}
    ctx, psi = state["ctx"], state["psi"]
    if kind == "apply":
        return ctx.apply_H(psi, prec=PREC[c["prec"]])
    if kind == "expm":
        out, k = ctx.expm(psi, c["dt"], prec=PREC[c["prec"]])
        return {"psi": out, "k": k}
    if kind == "fields":
        res = []
        for x in (psi, state["psi2"]):
            rho = ctx.density(x)
            vh, _ = ctx.hartree(rho)
            res.append({"rho": rho, "vh": vh, "vxc": ctx.xc(rho), "d": ctx.dipole(rho)})
        return res
    if kind == "steps":
        work = state["work"]
        work.copy_(psi)
        d = [ctx.init_propagation(work)]
        for n in range(c["steps"]):
            e = state["E"][n]
            d.append(np.array(ctx.magnus_step(work, c["dt"], e[:3], e[3:], prec=PREC[c["prec"]])["dipole"]))
        return {"psi": work, "d": np.stack(d)}
    E = state["E"]
    E.grad = None
    J = tdks.DipoleObjective.apply(E, ctx, psi, _weights(c), (0.0, 0.0, 1.0), c["dt"], c["ckpt"], 1e-12, 64,
                                   PREC[c["prec"]], 12)
    J.backward()
    return {"J": J.detach(), "grad": E.grad}


def work(case):
    """Bytes: inputs read once, outputs written once.  Flops: 36 (p+1)^4 + 24 (p+1)^3 per element, orbital and
    application (nine one-dimensional contractions of both components), 12 (p+1)^4 per element and orbital of
    a density; the applications of an exponential by the length of its Chebyshev expansion."""
    c, kind = case, case["kind"]
    if kind == "batch":
        w = [work(dict(q, kind="steps", steps=c["steps"])) for q in _batch_cases(c)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    P, ne = c["p"] + 1, c["nx"] * c["ny"] * c["nz"]
    vec, field = 16.0 * _n_int(c) * c["n_orb"], 8.0 * ne * P ** 3
    app = (36.0 * P ** 4 + 24.0 * P ** 3) * ne * c["n_orb"]
    dens = 12.0 * P ** 4 * ne * c["n_orb"]
    if kind == "apply":
        return {"bytes": 2 * vec + field, "flops": app}
    if kind == "fields":
        return {"bytes": 2 * (vec + 3 * field), "flops": 2 * dens}
    half = _half_width(c)
    terms = lambda t: t * half + 4.0 * (t * half) ** (1 / 3) + 6.0
    if kind == "expm":
        return {"bytes": 2 * vec + field, "flops": app * terms(c["dt"])}
    step = app * (terms(0.5 * c["dt"]) + terms(c["dt"])) + 2 * dens
    if kind == "steps":
        return {"bytes": 2 * vec, "flops": c["steps"] * step + dens}
    return {"bytes": vec + 96.0 * c["steps"], "flops": 4.0 * c["steps"] * step}


# ---- the same in plain torch, 64 bits ----------------------------------------------------------------------

def _gll(p):
    P = np.polynomial.legendre.Legendre.basis(p)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    for _ in range(3):                                   # Newton on the interior roots
        x[1:-1] -= P.deriv()(x[1:-1]) / P.deriv(2)(x[1:-1])
    x = 0.5 * (x - x[::-1])
    return x, 2.0 / (p * (p + 1) * P(x) ** 2)


def _lagrange(z, x):
    """Values [len(x), len(z)] of the Lagrange basis on z at x, and the derivatives."""
    n = len(z)
    val, der = np.ones((len(x), n)), np.zeros((len(x), n))
    for i in range(n):
        for m in range(n):
            if m != i:
                val[:, i] *= (x - z[m]) / (z[i] - z[m])
        for l in range(n):
            if l != i:
                t = np.full(len(x), 1.0 / (z[i] - z[l]))
                for m in range(n):
                    if m != i and m != l:
                        t *= (x - z[m]) / (z[i] - z[m])
                der[:, i] += t
    return val, der


class _Ref:
    def __init__(self, s):
        self.s, self.dev = s, torch.device("cuda" if torch.cuda.is_available() else "cpu")
        p, P = s["p"], s["p"] + 1
        t = lambda a: torch.as_tensor(a, dtype=F64, device=self.dev)
        xi, wl = _gll(p)
        eta, om = np.polynomial.legendre.leggauss(P)
        B, D = _lagrange(xi, eta)
        self.B, self.D, self.P = t(B), t(D), P
        K1, Mg = D.T @ np.diag(om) @ D, B.T @ np.diag(om) @ B
        self.n = [len(b) - 1 for b in s["br"]]
        self.idx, self.h, self.xq, self.wq, self.sm, self.node, self.eig, self.tmax = [], [], [], [], [], [], [], 0.0
        for b in s["br"]:
            n, h = len(b) - 1, np.diff(b)
            idx = np.arange(n)[:, None] * p + np.arange(P)[None, :]
            node = b[:-1, None] + 0.5 * (xi + 1) * h[:, None]
            mass, A, G = np.zeros(n * p + 1), np.zeros((n * p + 1,) * 2), np.zeros((n * p + 1,) * 2)
            x = np.zeros(n * p + 1)
            for e in range(n):
                i = idx[e]
                mass[i] += 0.5 * h[e] * wl
                x[i] = node[e]
                A[np.ix_(i, i)] += 2.0 / h[e] * K1
                G[np.ix_(i, i)] += 0.5 * h[e] * Mg
            A, G, sm = A[1:-1, 1:-1], G[1:-1, 1:-1], 1.0 / np.sqrt(mass[1:-1])
            Li = np.linalg.inv(np.linalg.cholesky(G))
            lam, Q = np.linalg.eigh(Li @ A @ Li.T)
            self.eig.append((t(lam), t(Li.T @ Q)))
            self.tmax += 0.5 * np.linalg.eigvalsh(sm[:, None] * A * sm[None, :]).max()
            self.idx.append(torch.as_tensor(idx, device=self.dev))
            self.h.append(t(h))
            self.xq.append(t(b[:-1, None] + 0.5 * (eta + 1) * h[:, None]))       # [n, q]
            self.wq.append(t(0.5 * h[:, None] * om[None, :]))                      # [n, q]
            self.sm.append(t(sm))
            self.node.append(t(x[1:-1]))
        self.Ni = [n * p - 1 for n in self.n]
        S = self.sm
        self.scale = (S[2][:, None, None] * S[1][None, :, None] * S[0][None, None, :]).reshape(-1)
        # weights at the Gauss points as [ez, qz, ey, qy, ex, qx]
        W = self.wq
        self.W = W[2][:, :, None, None, None, None] * W[1][None, None, :, :, None, None] * W[0]

    # element-local views [o, ez, c, ey, b, ex, a] <-> nodal [o, n_int]
    def gather(self, u):
        o = u.shape[0]
        u = torch.view_as_real(u) if u.is_complex() else u[..., None]
        q = u.shape[-1]
        u = u.reshape(o, self.Ni[2], self.Ni[1], self.Ni[0], q).permute(0, 4, 1, 2, 3)
        u = torch.nn.functional.pad(u, (1, 1, 1, 1, 1, 1))
        u = u[:, :, self.idx[2]][:, :, :, :, self.idx[1]][:, :, :, :, :, :, self.idx[0]]
        return u                                          # [o, re/im, ez, c, ey, b, ex, a]

    def scatter(self, r, cplx):
        o, q = r.shape[:2]
        for d, dim in ((2, 2), (1, 3), (0, 4)):          # axis by axis: (element, local) -> node
            n, P, p = self.n[d], self.P, self.P - 1
            shape = list(r.shape)
            out = torch.zeros(shape[:dim] + [n * p + 1] + shape[dim + 2:], dtype=r.dtype, device=r.device)
            r = out.index_add(dim, self.idx[d].reshape(-1), r.flatten(dim, dim + 1))
        r = r[:, :, 1:-1, 1:-1, 1:-1].reshape(o, q, -1)
        return torch.complex(r[:, 0], r[:, 1]) if cplx else r[:, 0]

    def along(self, M, u, d):
        dim = {0: 7, 1: 5, 2: 3}[d]
        return torch.movedim(torch.movedim(u, dim, -1) @ M.T, -1, dim)

    def to_q(self, u):
        u = self.gather(u)
        for d in (2, 1, 0):
            u = self.along(self.B, u, d)
        return u

    def from_q(self, r, cplx):
        for d in (2, 1, 0):
            r = self.along(self.B.T.contiguous(), r, d)
        return self.scatter(r, cplx)

    def field(self, f):                                    # [n_elem, q^3] -> [ez, qz, ey, qy, ex, qx]
        n, P = self.n, self.P
        return f.reshape(n[2], n[1], n[0], P, P, P).permute(0, 3, 1, 4, 2, 5)

    def unfield(self, f):
        return f.permute(0, 2, 4, 1, 3, 5).reshape(self.n[0] * self.n[1] * self.n[2], self.P ** 3)

    def coord(self, d):
        x = self.xq[d]
        return {0: x, 1: x[:, :, None, None], 2: x[:, :, None, None, None, None]}[d]

    def v_nuc(self):
        s, acc = self.s, 0.0
        for R, Z in zip(s["R"], s["Z"]):
            r = torch.sqrt(sum((self.coord(d) - float(R[d])) ** 2 for d in range(3)))
            if s["nuc"] == "soft":
                acc = acc - float(Z) / torch.sqrt(r * r + s["par"])
            elif s["nuc"] == "bare":
                acc = acc - float(Z) / r
            else:
                acc = acc - float(Z) * torch.erf(r / s["par"]) / r
        return self.unfield(acc)

    def apply(self, v, psi, kb=None):
        u = self.to_q(psi * self.scale)
        # kinetic form in the Gauss-point Lagrange basis: derivative of the interpolant along one axis
        Dg = self.D @ torch.linalg.inv(self.B)
        r = self.field(v) * self.W * u
        for d in range(3):
            ih = {0: 2.0 / self.h[0][:, None], 1: (2.0 / self.h[1])[:, None, None, None],
                  2: (2.0 / self.h[2])[:, None, None, None, None, None]}[d]
            r = r + 0.5 * self.along(Dg.T.contiguous(), ih * ih * self.W * self.along(Dg, u, d), d)
        out = self.from_q(r, True) * self.scale
        if kb is not None:
            out = out + ((psi @ kb[0]) * kb[1]) @ kb[0].T
        return out

    def projectors(self, a=1.0, b=0.8, c=(-2.0, -1.0)):
        cols, inv = [], []
        for R in self.s["R"]:
            x = [self.coord(d) - float(R[d]) for d in range(3)]
            r2 = sum(t * t for t in x)
            for l, Y in ((0, 1.0), (1, x[0]), (1, x[1]), (1, x[2])):
                u = torch.exp(-r2 / (2 * a * a)) * Y
                dv = c[l] * torch.exp(-r2 / (2 * b * b))
                cols.append((self.from_q((dv * u * self.W)[None, None], False)[0] * self.scale))
                inv.append(1.0 / (u * dv * u * self.W).sum())
        return torch.stack(cols, 1).to(C128), torch.stack(inv).to(C128)

    def expm(self, v, psi, t, kb=None):
        """exp(-i t Hbar) psi: Chebyshev expansion on an interval holding the spectrum (GLL mass >= Gauss mass)."""
        lo, hi = min(0.0, float(v.detach().min())), max(0.0, float(v.detach().max())) + self.tmax
        if kb is not None:
            ex = float(((kb[0].abs() ** 2).sum(0) * kb[1].abs()).sum())
            lo, hi = lo - ex, hi + ex
        c, R = 0.5 * (lo + hi), 0.5 * (hi - lo)
        z = t * R
        N = int(z + 14 * z ** (1 / 3) + 20)
        J = np.zeros(N + 42)                               # Miller's backward recurrence
        J[N + 40] = 1e-280
        for n in range(N + 40, 0, -1):
            J[n - 1] = 2.0 * n / z * J[n] - J[n + 1]
            if abs(J[n - 1]) > 1e250:
                J *= 1e-250
        J /= J[0] + 2 * J[2::2].sum()
        X = lambda u: (self.apply(v, u, kb) - c * u) / R
        a, b = psi, X(psi)
        out = J[0] * a - 2j * J[1] * b
        for n in range(2, N + 1):
            a, b = b, 2 * X(b) - a
            out = out + (2 * (-1j) ** n * J[n]) * b
        return out * np.exp(-1j * t * c)

    def density(self, psi):
        rho = 0.0
        for o in range(psi.shape[0]):
            u = self.to_q(psi[o:o + 1] * self.scale)
            rho = rho + 2.0 * (u[0] * u[0]).sum(0)
        return self.unfield(rho)

    def hartree(self, rho):
        b = 4 * math.pi * self.from_q((self.field(rho) * self.W)[None, None], False)[0]
        x = b.reshape(self.Ni[2], self.Ni[1], self.Ni[0])
        (lx, Sx), (ly, Sy), (lz, Sz) = self.eig
        x = torch.einsum("kji,ia,jb,kc->cba", x, Sx, Sy, Sz)
        x = x / (lz[:, None, None] + ly[None, :, None] + lx[None, None, :])
        phi = torch.einsum("cba,ia,jb,kc->kji", x, Sx, Sy, Sz).reshape(1, -1)
        return self.unfield(self.to_q(phi)[0, 0])

    @staticmethod
    def xc(rho):
        """Perdew-Zunger 1981, unpolarized; 0 below 1e-14."""
        ok = rho >= 1e-14
        r = torch.where(ok, rho, torch.ones_like(rho))
        rs = (3.0 / (4.0 * math.pi * r)) ** (1 / 3)
        sq = rs.sqrt()
        den = 1.0 + 1.0529 * sq + 0.3334 * rs
        low = -0.1423 / den * (1 + 7 / 6 * 1.0529 * sq + 4 / 3 * 0.3334 * rs) / den
        lr = rs.log()
        high = 0.0311 * lr + (-0.048 - 0.0311 / 3) + 2 / 3 * 0.0020 * rs * lr + (2 * -0.0116 - 0.0020) / 3 * rs
        return torch.where(ok, -(3.0 * r / math.pi) ** (1 / 3) + torch.where(rs >= 1, low, high), torch.zeros_like(rho))

    def dipole(self, rho):
        f = self.field(rho) * self.W
        return torch.stack([(f * self.coord(d)).sum() for d in range(3)])

    def field_term(self, E):
        return self.unfield(sum(E[d] * self.coord(d) for d in range(3)) + torch.zeros_like(self.W))

    def steps(self, psi, dt, E):
        """Predictor-corrector steps with field samples E [n, 6]: (psi, dipoles [n + 1, 3])."""
        hxc = lambda rho: self.hartree(rho) + self.xc(rho)
        vn = self.v_nuc()
        rho = self.density(psi)
        h1 = h2 = hxc(rho)
        d = [self.dipole(rho)]
        for e in E:
            half = self.expm(vn + 1.25 * h1 - 0.25 * h2 - self.field_term(e[:3]), psi, 0.5 * dt)
            psi = self.expm(vn + hxc(self.density(half)) - self.field_term(e[3:]), psi, dt)
            rho = self.density(psi)
            h1, h2 = hxc(rho), h1
            d.append(self.dipole(rho))
        return psi, torch.stack(d)

    def kick(self, psi, kappa):
        return psi * torch.exp(-1j * kappa * self.node[0]).repeat(self.Ni[1] * self.Ni[2])


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "batch":
        d, psi, d0 = [], [], []
        for k, q in enumerate(_batch_cases(c)):
            ref = _Ref(_system(q, np.random.default_rng([seed, k])))
            with torch.no_grad():
                x, dk = ref.steps(_orbitals(q, seed + 1000 * k), q["dt"], torch.zeros(c["steps"], 6, dtype=F64))
            psi.append(x)
            d0.append(dk[0])
            d.append(dk[1:])
        return {"d0": torch.stack(d0), "d": torch.stack(d, 1), "psi": psi}
    s = _system(c, np.random.default_rng([seed, 0]))
    ref, psi = _Ref(s), _orbitals(c, seed)
    if kind == "gradient":
        E = torch.from_numpy(_fields_E(c, seed)).to(ref.dev).requires_grad_(True)
        d = ref.steps(psi, c["dt"], E)[1]
        J = (torch.as_tensor(_weights(c), device=ref.dev) * d[:, 2] ** 2).sum()
        J.backward()
        return {"J": J.detach(), "grad": E.grad}
    with torch.no_grad():
        if kind == "apply":
            return ref.apply(_potential(c, s, seed), psi)
        if kind == "expm":
            return {"psi": ref.expm(_potential(c, s, seed), psi, c["dt"], ref.projectors() if c["kb"] else None),
                    "k": None}
        if kind == "fields":
            out = []
            for x in (psi, _orbitals(c, seed + 500)):
                rho = ref.density(x)
                out.append({"rho": rho, "vh": ref.hartree(rho), "vxc": ref.xc(rho), "d": ref.dipole(rho)})
            return out
        x, d = ref.steps(ref.kick(psi, KICK), c["dt"], torch.from_numpy(_fields_E(c, seed)).to(ref.dev))
        return {"psi": x, "d": d}

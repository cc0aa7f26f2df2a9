"""FP64 Hbar psi and density (csrc/hbar_fx.cu) on orbitals that fall off steeply inside an
element, against extended precision (numpy's long double), entry by entry.

Bounds: what FP64 arithmetic of the same chain may lose.  An entry of Hbar psi is a sum over
products of the tables, the geometry and psi; its error is at most the number of roundings
that a term passes, times 2^-53, times the sum of the terms' magnitudes (the chain with every
factor replaced by its magnitude).  A term passes 9 roundings of the Loewdin scales on either
side, 3 of the input's scaling, 7 of the geometry and the tables, 2 (p + 1) of the nine
contractions' sums on average, 8 of the gather and 3 of its scaling."""
import numpy as np
import pytest

import synth
from oracle.mesh import Mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LD = np.longdouble
U = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1810_13130_gb300.build import build
    build()


def _legendre(n, x):
    a, b = np.ones_like(x), x
    for k in range(1, n):
        a, b = b, ((2 * k + 1) * x * b - k * a) / LD(k + 1)
    return b, n * (a - x * b) / (1 - x * x)


def _tables(p):
    """GLL nodes and weights, Gauss weights, values and derivatives of the GLL Lagrange basis at the Gauss points."""
    t = -np.cos(LD(np.pi) * np.arange(1, p).astype(LD) / p)
    e = -np.cos(LD(np.pi) * (np.arange(p + 1).astype(LD) + LD(0.75)) / (p + LD(1.5)))
    for _ in range(60):
        P, d = _legendre(p, t)
        t = t - d / ((2 * t * d - LD(p * (p + 1)) * P) / (1 - t * t))
        P, d = _legendre(p + 1, e)
        e = e - P / d
    xi = np.concatenate([[LD(-1)], t, [LD(1)]])
    Pn = np.concatenate([[LD((-1) ** p)], _legendre(p, t)[0] if p > 1 else [], [LD(1)]])
    om = 2 / ((1 - e * e) * _legendre(p + 1, e)[1] ** 2)
    B, D = np.ones((p + 1, p + 1), LD), np.zeros((p + 1, p + 1), LD)
    for i in range(p + 1):
        for m in range(p + 1):
            if m != i:
                B[:, i] *= (e - xi[m]) / (xi[i] - xi[m])
                s = np.full(p + 1, 1 / (xi[i] - xi[m]))
                for l in range(p + 1):
                    if l not in (i, m):
                        s *= (e - xi[l]) / (xi[i] - xi[l])
                D[:, i] += s
    return xi, 2 / (p * (p + 1) * Pn ** 2), om, B, D


class Ref:
    """Axis matrices over all elements: interpolation to the Gauss points, Gauss-point stiffness, scales."""

    def __init__(self, breaks, p):
        xi, wl, om, B, D = _tables(p)
        Dg = D @ np.linalg.inv(B.astype(float)).astype(LD)           # refined: D = Dg B
        for _ in range(3):
            Dg = Dg + (D - Dg @ B) @ np.linalg.inv(B.astype(float)).astype(LD)
        self.ax = []
        for b in breaks:
            n, P = len(b) - 1, p + 1
            I, K = np.zeros((n * P, n * p + 1), LD), np.zeros((n * P, n * P), LD)
            mass, w, x = np.zeros(n * p + 1, LD), np.zeros(n * P, LD), np.zeros(n * p + 1)
            for e in range(n):
                h, q, c = LD(b[e + 1]) - LD(b[e]), slice(e * P, e * P + P), slice(e * p, e * p + P)
                I[q, c], w[q] = B, om * h / 2
                K[q, q] = (Dg.T * om) @ Dg * 2 / h
                mass[c] += wl * h / 2
                x[c] = (LD(b[e]) + (xi + 1) * h / 2).astype(float)
            self.ax.append((I[:, 1:-1], K, w, 1 / np.sqrt(mass[1:-1]), x[1:-1]))

    def each(self, u, M, d):
        return np.moveaxis(np.tensordot(M, u, axes=(1, 2 - d)), 0, 2 - d)

    def _all(self, u, k, mag, tr=False):
        for d in range(3):
            M = self.ax[d][k].T if tr else self.ax[d][k]
            u = self.each(u, abs(M) if mag else M, d)
        return u

    def outer(self, k):
        a = [self.ax[d][k] for d in range(3)]
        return a[2][:, None, None] * a[1][None, :, None] * a[0][None, None, :]

    def to_q(self, psi, mag=False):
        return self._all(psi.astype(LD) * self.outer(3), 0, mag)

    def apply(self, v, psi, mag=False):
        u = self.to_q(psi, mag)
        r = (abs(v) if mag else v) * self.outer(2) * u
        for d in range(3):
            W = [self.ax[e][2] if e != d else np.ones_like(self.ax[e][2]) for e in range(3)]
            t = self.each(u, abs(self.ax[d][1]) if mag else self.ax[d][1], d) / 2
            r = r + t * W[2][:, None, None] * W[1][None, :, None] * W[0][None, None, :]
        return self._all(r, 0, mag, tr=True) * self.outer(3)


def _steep(ref, p, decay, n_orb, seed):
    """exp(-decay r / h) around an interior node, real and imaginary parts of their own; the sign of every entry too."""
    rng = np.random.default_rng(seed)
    x = [ref.ax[d][4] for d in range(3)]
    out = []
    for o in range(n_orb):
        c = [t[min(len(t) - 1, o * (p // 2))] for t in x]
        h = [np.ptp(t) / max(1, len(t) - 1) * p if len(t) > 1 else 1.0 for t in x]
        r = np.sqrt(((x[2] - c[2]) / h[2])[:, None, None] ** 2 + ((x[1] - c[1]) / h[1])[None, :, None] ** 2 +
                    ((x[0] - c[0]) / h[0])[None, None, :] ** 2)
        f = np.exp(-decay * r)
        out.append(f * rng.uniform(0.5, 1, f.shape) + 1j * f * (1 if o % 2 else rng.uniform(-1, 1, f.shape)))
    return np.array(out)


def _setup(p, n, n_orb):
    from paper_1810_13130_gb300 import tdks
    cfg = synth.small_config(*n, p=p, n_orb=n_orb, graded=True, seed=97)
    return tdks.Context.from_config(cfg), Ref((cfg.X, cfg.Y, cfg.Z), p), Mesh.from_config(cfg)


def _grid(f, n, P):      # [n_elem, P^3] field -> [z, y, x] over all Gauss points
    return f.reshape(n[2], n[1], n[0], P, P, P).transpose(0, 3, 1, 4, 2, 5).reshape(n[2] * P, n[1] * P, n[0] * P)


@pytest.mark.parametrize("decay", [0.0, 8.0, 20.0])
@pytest.mark.parametrize("p,n", [(2, (3, 2, 2)), (4, (2, 1, 2)), (5, (1, 2, 1)), (6, (1, 1, 2)), (8, (2, 1, 1))])
def test_apply(p, n, decay):
    ctx, ref, m = _setup(p, n, 3)
    rng = np.random.default_rng(98)
    v = -20.0 * np.exp(3 * rng.uniform(-1, 1, (m.n_elem, (p + 1) ** 3)))
    psi = _steep(ref, p, decay, 3, 99)
    ctx.set_potential(torch.from_numpy(v).cuda())
    out = ctx.apply_H(torch.from_numpy(psi.reshape(3, -1)).cuda()).cpu().numpy().reshape(psi.shape)
    vq = _grid(v, n, p + 1)
    bound = (18 + 3 + 7 + 2 * (p + 1) + 11) * U
    for o in range(3):
        for part, got in ((psi[o].real, out[o].real), (psi[o].imag, out[o].imag)):
            err = abs(got - ref.apply(vq, part))
            assert (err <= bound * ref.apply(vq, abs(part), mag=True)).all()
    ctx.close()


@pytest.mark.parametrize("decay", [0.0, 8.0, 20.0])
@pytest.mark.parametrize("p,n", [(3, (2, 2, 1)), (4, (2, 1, 2)), (6, (1, 1, 2)), (8, (2, 1, 1))])
def test_density(p, n, decay):
    ctx, ref, m = _setup(p, n, 2)
    psi = _steep(ref, p, decay, 2, 96)
    rho = _grid(ctx.density(torch.from_numpy(psi.reshape(2, -1)).cuda()).cpu().numpy(), n, p + 1)
    # per part: 9 roundings of the scales, 3 of the input, p + 1 of the sums, twice in the square;
    # occupations, weights and the sum over parts and orbitals
    c = (9 + 3 + p + 1) * U
    exact, bound = 0, 0
    for o in range(2):
        for part in (psi[o].real, psi[o].imag):
            u, mag = ref.to_q(part), ref.to_q(abs(part), mag=True)
            exact = exact + 2 * u * u
            bound = bound + 4 * c * abs(u) * mag + 2 * (c * mag) ** 2
    assert (abs(rho - exact) <= bound + 12 * U * exact).all()
    ctx.close()


@pytest.mark.parametrize("p,n,n_orb", [(1, (3, 2, 2), 1), (4, (2, 1, 2), 1), (4, (4, 4, 5), 8), (7, (2, 2, 2), 3)])
def test_parts_are_independent(p, n, n_orb):
    """Hbar is real: the parts of a complex vector have their own exponents, however far apart they lie."""
    ctx, ref, m = _setup(p, n, n_orb)
    v = synth.random_potential(m.n_elem * m.nq ** 3, seed=95).reshape(m.n_elem, -1)
    ctx.set_potential(torch.from_numpy(v).cuda())
    a = torch.from_numpy(synth.random_psi(n_orb, m.N_int, seed=94).real.copy()).cuda()
    b = torch.from_numpy(synth.random_psi(n_orb, m.N_int, seed=93).real.copy()).cuda()
    zero = torch.zeros_like(a)
    Ha, Hb = (ctx.apply_H(torch.complex(x, zero).contiguous()) for x in (a, b))
    assert not Ha.imag.any() and not Hb.imag.any()
    for k in (0, 40, 200):
        out = ctx.apply_H(torch.complex(a, b * 2.0 ** -k).contiguous())
        assert torch.equal(out.real, Ha.real) and torch.equal(out.imag, Hb.real * 2.0 ** -k), k
        out = ctx.apply_H(torch.complex(a * 2.0 ** -k, b).contiguous())
        assert torch.equal(out.real, Ha.real * 2.0 ** -k) and torch.equal(out.imag, Hb.real), k
    ctx.close()


@pytest.mark.parametrize("decay", [0.0, 8.0, 20.0])
@pytest.mark.parametrize("p,n", [(3, (2, 2, 1)), (4, (2, 1, 2)), (6, (1, 1, 2)), (7, (2, 1, 1)), (8, (2, 1, 1))])
def test_first_lanczos_coefficient(p, n, decay):
    """alpha_0 = <psi|Hbar|psi> / <psi|psi> is the phase per time of a one-dimensional Krylov exponential."""
    ctx, ref, m = _setup(p, n, 2)
    rng = np.random.default_rng(92)
    v = -20.0 * np.exp(3 * rng.uniform(-1, 1, (m.n_elem, (p + 1) ** 3)))
    psi = _steep(ref, p, decay, 2, 91)
    ctx.set_potential(torch.from_numpy(v).cuda())
    vq = _grid(v, n, p + 1)
    # the roundings of an entry of Hbar psi (test_apply) and 2 of the sums, for the larger part;
    # the angle of a component comes back within 4 roundings of 1
    bound = (18 + 3 + 7 + 2 * (p + 1) + 11 + 2) * U
    for o in range(2):
        x = [psi[o].real.astype(LD), psi[o].imag.astype(LD)]
        nrm = sum((t * t).sum() for t in x)
        alpha = sum((t * ref.apply(vq, t)).sum() for t in x) / nrm
        mag = sum((abs(t) * ref.apply(vq, abs(t), mag=True)).sum() for t in x) / nrm
        tau = float(1 / mag)
        out, _ = ctx.expm(torch.from_numpy(psi[o:o + 1].reshape(1, -1).copy()).cuda(), tau, tol=1e30, k_max=1)
        got = -np.angle(np.vdot(psi[o].ravel(), out.cpu().numpy().ravel())) / tau
        assert abs(got - alpha) <= bound * mag + 4 * U / tau
    ctx.close()

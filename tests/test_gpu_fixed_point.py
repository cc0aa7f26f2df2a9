"""The fixed-point element kernel of the FP64 Hbar application (csrc/hbar_fx.cu) at the
edges of its range: block exponents near both ends of FP64, zero blocks, non-finite inputs
and potentials, and the launch shapes of small and large calls.

Every element and orbital carries its own power-of-two exponent, so scaling the input by a
power of two scales the result exactly, whatever the launch shape."""
import numpy as np
import pytest

import synth
from oracle import hamiltonian as ham
from oracle.mesh import Mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1810_13130_gb300.build import build
    build()


def _setup(p, n, n_orb, graded=True):
    from paper_1810_13130_gb300 import tdks
    cfg = synth.small_config(*n, p=p, n_orb=n_orb, graded=graded, seed=51 + p)
    m = Mesh.from_config(cfg)
    v = synth.random_potential(m.n_elem * m.nq ** 3, seed=60 + p).reshape(m.n_elem, -1)
    psi = synth.random_psi(n_orb, m.N_int, seed=70 + p)
    return tdks.Context.from_config(cfg), m, v, psi


# the smallest mesh of a degree, uneven meshes, one CTA and several
SHAPES = [(1, (2, 2, 2)), (2, (1, 2, 1)), (3, (5, 3, 2)), (4, (1, 1, 1)), (5, (2, 3, 4)), (6, (3, 1, 2)), (7, (2, 2, 1)),
          (8, (2, 1, 3))]


@pytest.mark.parametrize("p,n", SHAPES)
def test_power_of_two_scaling_is_exact(p, n):
    ctx, m, v, psi = _setup(p, n, 3)
    psi[1] = 0.0
    ctx.set_potential(torch.from_numpy(v).cuda())
    base = ctx.apply_H(torch.from_numpy(psi).cuda()).cpu().numpy()
    ref = ham.apply_H(m, v, psi)
    # FP64 rounds each of ~3 (p + 1) products of a contraction chain of 7 to 2^-53 of terms no
    # larger than |K| |psi|; 1e-13 of the largest entry covers that for these degrees
    assert np.abs(base - ref).max() <= 1e-13 * np.abs(ref).max()
    assert not base[1].any()
    for k in (-880, -300, 500, 900):
        out = ctx.apply_H(torch.from_numpy(psi * 2.0 ** k).cuda()).cpu().numpy()
        assert np.array_equal(out, base * 2.0 ** k), k
    ctx.close()


@pytest.mark.parametrize("p,n", [(2, (4, 3, 3)), (6, (3, 3, 3)), (8, (2, 2, 2))])
def test_launch_shapes_agree(p, n):
    """One orbital (few elements per CTA) and 24 orbitals (full CTAs, several orbitals each)."""
    ctx, m, v, psi = _setup(p, n, 24)
    ctx.set_potential(torch.from_numpy(v).cuda())
    g = torch.from_numpy(psi).cuda()
    full = ctx.apply_H(g)
    for tile in (1, 5, 24):
        ctx.set_apply_tile(tile)
        assert torch.equal(ctx.apply_H(g), full)
    ctx.set_apply_tile(0)
    for o in (0, 23):
        assert torch.equal(ctx.apply_H(g[o:o + 1].contiguous())[0], full[o])
    ctx.close()


@pytest.mark.parametrize("p", [3, 6])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values_stay_in_their_elements(p, bad):
    ctx, m, v, psi = _setup(p, (4, 2, 2), 2)
    Ni = tuple(m.Ni)
    ctx.set_potential(torch.from_numpy(v).cuda())
    clean = ctx.apply_H(torch.from_numpy(psi).cuda()).cpu().numpy().reshape(2, Ni[2], Ni[1], Ni[0])
    # an interior node of the first element (x index p // 2): its element's nodes are lost
    x = psi.copy().reshape(2, Ni[2], Ni[1], Ni[0])
    x[1, p // 2 - 1, p // 2 - 1, p // 2 - 1] = bad
    out = ctx.apply_H(torch.from_numpy(x.reshape(2, -1)).cuda()).cpu().numpy().reshape(clean.shape)
    hit = np.zeros(clean.shape, bool)
    hit[1, :p, :p, :p] = True
    assert np.isnan(out[hit]).all() and np.array_equal(out[~hit], clean[~hit])
    # a potential value of the last element
    w = v.copy()
    w[-1, 3] = bad
    ctx.set_potential(torch.from_numpy(w).cuda())
    out = ctx.apply_H(torch.from_numpy(psi).cuda()).cpu().numpy().reshape(clean.shape)
    hit[:] = False
    hit[:, p - 1:, p - 1:, 3 * p - 1:] = True
    assert np.isnan(out[hit]).all() and np.array_equal(out[~hit], clean[~hit])
    ctx.close()


@pytest.mark.parametrize("p,n", SHAPES)
def test_density(p, n):
    """The FP64 density (Eq. 2): three contractions, squares summed over the orbitals."""
    ctx, m, v, psi = _setup(p, n, 3)
    ref = ham.density(m, psi, [2.0] * 3).ravel()
    rho = ctx.density(torch.from_numpy(psi).cuda()).cpu().numpy().ravel()
    # the oracle rounds three FP64 contractions of p + 1 terms: within 1e-13 of the largest value
    assert np.abs(rho - ref).max() <= 1e-13 * ref.max()
    for k in (-400, 300):
        out = ctx.density(torch.from_numpy(psi * 2.0 ** k).cuda()).cpu().numpy().ravel()
        assert np.array_equal(out, rho * 4.0 ** k), k
    # a non-finite entry loses its element's density and no other
    x = psi.copy()
    x[1, 0] = np.nan
    out = ctx.density(torch.from_numpy(x).cuda()).cpu().numpy().ravel()
    nq = m.nq ** 3
    own = 1 if p > 1 else 8     # (p = 1: the first interior node belongs to eight elements)
    assert np.isnan(out[:nq]).all() and np.isnan(out).sum() == own * nq
    assert np.array_equal(out[8 * nq:], rho[8 * nq:]) if p == 1 else np.array_equal(out[nq:], rho[nq:])
    ctx.close()

"""Captured Lanczos loops (csrc/krylov.cu) when the buffers behind them change between two
exponentials: projectors replaced by others, a Krylov basis of another length, the adjoint's
second basis.  The host-driven loop of a fresh context runs the same kernels in the same
order, so results are equal to the bit."""
import numpy as np
import pytest

import synth
from oracle.mesh import Mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1810_13130_gb300.build import build
    build()


def _context(cfg, v, loop):
    from paper_1810_13130_gb300 import tdks
    ctx = tdks.Context.from_config(cfg)
    ctx.set_cg(1e-13)
    ctx.set_potential(torch.from_numpy(v).cuda())
    ctx.set_device_loop(loop)
    return ctx


# positions, projectors per atom; the same count at other places is the likeliest to meet
# the addresses of the one before
KB = [(np.array([[0.3, -0.2, 0.1], [-2.0, 1.5, 0.7]]), 1), (np.array([[-1.1, 0.9, -0.4], [2.0, -1.5, 1.7]]), 1),
      (np.array([[0.5, 0.5, -0.5], [1.0, -2.0, 0.0], [-1.5, 0.3, 2.2]]), 0), (np.zeros((0, 3)), 1),
      (np.array([[2.4, 0.1, -1.0]]), 1)]


def test_projectors_replaced_between_exponentials():
    cfg = synth.small_config(4, 3, 3, p=4, n_orb=3, seed=61)
    m = Mesh.from_config(cfg)
    v = synth.random_potential(m.n_elem * m.nq ** 3, seed=62).reshape(m.n_elem, -1)
    g = torch.from_numpy(synth.random_psi(3, m.N_int, seed=63)).cuda()
    ctx = _context(cfg, v, 1)
    for R, lmax in KB + KB[:2]:
        ctx.set_kb(R, lmax=lmax)
        for _ in range(2):
            out, k = ctx.expm(g, 0.05)
        fresh = _context(cfg, v, 0)
        fresh.set_kb(R, lmax=lmax)
        ref, kref = fresh.expm(g, 0.05)
        assert k == kref and torch.equal(out, ref)
        fresh.close()
    ctx.close()


def test_bases_replaced_between_exponentials():
    cfg = synth.small_config(3, 3, 3, p=4, n_orb=2, seed=64)
    m = Mesh.from_config(cfg)
    v = synth.random_potential(m.n_elem * m.nq ** 3, seed=65).reshape(m.n_elem, -1)
    psi = torch.from_numpy(synth.smooth_orbitals(tuple(m.Ni), 2, seed=66)).cuda()
    E = 1e-2 * np.random.default_rng(67).standard_normal((2, 6))

    def gradient(ctx, k_max):
        ctx.objective_forward(psi, E, np.ones(3), (0.0, 0.0, 1.0), 0.02, 2, 1e-11, k_max)
        return ctx.objective_backward(6)

    ctx = _context(cfg, v, 1)
    for k_max in (40, 64, 40, 48):          # the second basis may take the place that the first left
        got = gradient(ctx, k_max)
        ctx.set_potential(torch.from_numpy(v).cuda())
        out, k = ctx.expm(psi, 0.02, k_max=k_max + 5)
        fresh = _context(cfg, v, 0)
        ref, kref = fresh.expm(psi, 0.02, k_max=k_max + 5)
        assert k == kref and torch.equal(out, ref)
        assert np.array_equal(got, gradient(fresh, k_max))
        fresh.close()
    ctx.close()

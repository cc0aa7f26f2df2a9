"""The nonlocal projection and gather (csrc/kb.cu) at the edges of their work splits: boxes
shorter and longer than one projection chunk, one projector per atom and four, an atom
whose box is cut by the boundary, and orbital counts around the gather's block of four,
also beyond the system's own count."""
import numpy as np
import pytest

import synth
from oracle import hamiltonian as ham
from oracle.kb import KleinmanBylander
from oracle.mesh import Mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1810_13130_gb300.build import build
    build()


@pytest.mark.parametrize("p,n,lmax", [(2, (3, 2, 2), 1), (5, (4, 3, 3), 0), (6, (4, 4, 3), 1)])
def test_projection_shapes_match_oracle(p, n, lmax):
    from paper_1810_13130_gb300 import tdks
    cfg = synth.small_config(*n, p=p, n_orb=2, seed=81)
    m = Mesh.from_config(cfg)
    kp = synth.KBParams()
    R = np.array([[0.3, -0.2, 0.1], [-2.0, 1.5, 0.7], [5.6, -5.5, 5.2]])
    kb = KleinmanBylander(m, R, kp.a, kp.b, kp.c, lmax=lmax)
    ctx = tdks.Context.from_config(cfg)
    ctx.set_kb(R, kp.a, kp.b, kp.c, lmax)
    v = synth.random_potential(m.n_elem * m.nq ** 3, seed=82).reshape(m.n_elem, -1)
    ctx.set_potential(torch.from_numpy(v).cuda())
    for n_orb in (1, 2, 4, 5, 9):
        psi = synth.random_psi(n_orb, m.N_int, seed=83 + n_orb)
        ref = ham.apply_H(m, v, psi) + kb.apply(psi)
        got = ctx.apply_H(torch.from_numpy(psi).cuda()).cpu().numpy()
        # the bound of the projector-free application, test_gpu_parity
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max(), n_orb
    ctx.close()

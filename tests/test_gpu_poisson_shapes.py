"""The Poisson preconditioner's products (csrc/poisson.cu) at the edges of their tiles (16, 32)
and of the fixed-point form (255 terms; longer axes are FP64): axes of 1 to 263 nodes."""
import numpy as np
import pytest

import synth
from oracle import hamiltonian as ham, poisson
from oracle.mesh import Mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1810_13130_gb300.build import build
    build()


# interior nodes per axis: p n - 1
@pytest.mark.parametrize("p,n", [(2, (1, 1, 1)), (2, (8, 9, 1)), (3, (5, 6, 11)), (2, (16, 17, 3)), (8, (4, 2, 4)),
                                 (4, (64, 1, 1)), (4, (1, 64, 2)), (8, (1, 1, 33)), (4, (65, 2, 1))])
def test_preconditioner_is_the_inverse(p, n):
    from paper_1810_13130_gb300 import tdks
    cfg = synth.small_config(*n, p=p, n_orb=1, graded=True, seed=80 + p)
    m = Mesh.from_config(cfg)
    rho = ham.density(m, synth.random_psi(1, m.N_int, seed=81), cfg.occ)
    ctx = tdks.Context.from_config(cfg)
    ctx.set_cg(1e-10, 5000, 0)
    # the fast diagonalization is the inverse up to rounding: a wrong entry in any product
    # would leave a residual that takes CG more than a second iteration.  The condition number
    # of these stiffness matrices is below 1e5, so a residual of 1e-10 |b| is within 1e-5.
    ref, _, _ = poisson.hartree(m, rho, tol=1e-13)
    for k in (0, 100):   # values of any scale: the exponents are the rows' and columns' own
        vh, it = ctx.hartree(torch.from_numpy(np.ascontiguousarray(rho) * 2.0 ** k).cuda())
        assert it <= 2
        assert np.linalg.norm(vh.cpu().numpy().ravel() * 2.0 ** -k - ref.ravel()) <= 1e-5 * np.linalg.norm(ref)
    ctx.close()

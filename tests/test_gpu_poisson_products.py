"""The Poisson preconditioner's products (csrc/poisson.cu), seen through the residual they leave:
with products as accurate as FP64 the fast diagonalization takes these solves to 1e-12 in one CG
iteration (long axes: to 1e-13 in two), as it does with FP64 products throughout; products a
hundred times less accurate need another.  Axes at the edges of the tiles (16, 32), of the depth
tile and of the fixed-point form (16 to 255 nodes; the others are FP64)."""
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


# interior nodes per axis: p n - 1
@pytest.mark.parametrize("p,n,tol,its", [(2, (1, 1, 1), 1e-12, 1), (2, (8, 9, 1), 1e-12, 1), (1, (17, 16, 18), 1e-12, 1),
                                         (4, (4, 4, 4), 1e-12, 1), (6, (3, 3, 3), 1e-12, 1), (8, (4, 4, 5), 1e-12, 1),
                                         (3, (11, 5, 5), 1e-12, 1), (2, (17, 17, 16), 1e-12, 1),
                                         (8, (32, 1, 2), 1e-13, 2), (1, (256, 18, 17), 1e-13, 2), (1, (257, 3, 3), 1e-13, 2)])
def test_iterations_of_fp64_products(p, n, tol, its):
    from paper_1810_13130_gb300 import tdks
    for graded in (False, True):
        cfg = synth.small_config(*n, p=p, n_orb=1, graded=graded, seed=80 + p)
        m = Mesh.from_config(cfg)
        rho = ham.density(m, synth.random_psi(1, m.N_int, seed=81), cfg.occ)
        ctx = tdks.Context.from_config(cfg)
        ctx.set_cg(tol, 5000, 0)
        _, it = ctx.hartree(torch.from_numpy(np.ascontiguousarray(rho)).cuda())
        assert it <= its
        ctx.close()

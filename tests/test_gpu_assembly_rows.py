"""The FP64 gather with many rows per block (csrc/elements.cu): nodes on element faces after
those inside, row scales formed once per row; x rows shorter and longer than a block."""
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


# 64 orbitals: 128 blocks per orbital, more than four rows per block and row slot
@pytest.mark.parametrize("p,n", [(1, (130, 24, 24)), (2, (50, 12, 12)), (3, (43, 8, 8)), (4, (12, 12, 12))])
def test_many_rows_per_block(p, n):
    from paper_1810_13130_gb300 import tdks
    cfg = synth.small_config(*n, p=p, n_orb=64, graded=True, seed=90 + p)
    m = Mesh.from_config(cfg)
    v = synth.random_potential(m.n_elem * m.nq ** 3, seed=91).reshape(m.n_elem, -1)
    psi = synth.random_psi(64, m.N_int, seed=92)
    ctx = tdks.Context.from_config(cfg)
    ctx.set_potential(torch.from_numpy(v).cuda())
    g = torch.from_numpy(psi).cuda()
    out = ctx.apply_H(g)
    # one orbital takes a few rows per block: the same contributions in the same order
    for o in (0, 63):
        assert torch.equal(ctx.apply_H(g[o:o + 1].contiguous())[0], out[o])
    ref = ham.apply_H(m, v, psi[:1])
    # within 1e-13 of the largest entry: FP64 rounding of the oracle's contraction chain
    assert np.abs(out[:1].cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()
    ctx.close()

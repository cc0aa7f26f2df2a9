"""The exponential of a set with one orbital that fails: the call raises, the other orbitals hold
their results and the failed one holds its input, whether the result has its own buffer or not."""
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


@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("loop", [0, 1])
@pytest.mark.parametrize("in_place", [False, True])
def test_failed_orbital_keeps_its_input(prec, loop, in_place):
    from paper_1810_13130_gb300 import tdks
    cfg = synth.small_config(3, 2, 2, p=4, n_orb=3, seed=71)
    m = Mesh.from_config(cfg)
    v = synth.random_potential(m.n_elem * m.nq ** 3, seed=72).reshape(m.n_elem, -1)
    ctx = tdks.Context.from_config(cfg)
    ctx.set_device_loop(loop)
    ctx.set_potential(torch.from_numpy(v).cuda())
    good = torch.from_numpy(synth.random_psi(3, m.N_int, seed=73)).cuda()
    ref, _ = ctx.expm(good, 0.02, prec=prec)
    psi = good.clone()
    psi[1, 5] = float("nan")          # its norm is not finite: no recurrence starts
    out = psi.clone() if in_place else torch.full_like(psi, 7.0)
    with pytest.raises(tdks.TDKSError):
        ctx.expm(out if in_place else psi, 0.02, prec=prec, out=out)
    bits = lambda x: torch.view_as_real(x).contiguous().view(torch.int64)
    assert torch.equal(bits(out[1]), bits(psi[1]))
    for o in (0, 2):
        assert torch.equal(out[o], ref[o])
    ctx.close()

"""tdks_batch_set_kb with arguments that are refused, after a step with projectors: the old
projectors are gone, as with tdks_set_kb, and so is the captured step that held their buffers."""
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


@pytest.mark.parametrize("bad", [dict(lmax=2), dict(a=-1.0)])
def test_refused_projectors_leave_none(bad):
    from paper_1810_13130_gb300 import tdks
    cfgs = synth.small_batch()[:3]
    psi = [synth.random_psi(c.n_orb, Mesh.from_config(c).N_int, seed=40 + k) for k, c in enumerate(cfgs)]
    R = np.array([[0.3, -0.2, 0.1], [-2.1, 1.4, 0.9]])

    def start(b):
        for k, p in enumerate(psi):
            b.set_orbitals(k, torch.from_numpy(p).cuda())
        b.init()

    dts = [c.dt for c in cfgs]
    b, plain = tdks.Batch(cfgs, dts), tdks.Batch(cfgs, dts)
    b.set_kb(0, R)
    start(b)
    b.steps(1)
    with pytest.raises(tdks.TDKSError):
        b.set_kb(0, R, **bad)
    start(b)
    start(plain)
    # (the Poisson solves start from other guesses: equal to their tolerance)
    np.testing.assert_allclose(b.steps(2), plain.steps(2), rtol=1e-9, atol=1e-12)

"""Block solves with many MR steps: what is left of the residual is the rounding
of the fields and of one application of the operator, however many steps there
were.  One cycle from zero solves every block of the first colour on the given
source, so eta - D psi on such a block (psi zero elsewhere, D the oracle's in FP64)
is the block's residual.
"""
import numpy as np
import pytest

from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# links, clover term, solution and every term of the sums are rounded once, each to a
# unit u of numbers whose squares add up to a few |eta|^2: 8 u |eta|
TOL = {"f64": 8 * 2.0 ** -53, "f32": 8 * 2.0 ** -24, "f16": 8 * 2.0 ** -11, "bf16": 8 * 2.0 ** -8}


@pytest.mark.parametrize("spread,m0", [(0.5, 0.0), (0.9, -0.2), (0.5, -0.3)])
@pytest.mark.parametrize("prec,block", [("f64", (4, 4, 4, 2)), ("f32", (4, 4, 4, 4)), ("f32", (2, 4, 4, 8)),
                                        ("f16", (4, 4, 4, 4)), ("bf16", (4, 4, 4, 4))], ids=str)
def test_many_steps(orc, prec, block, spread, m0):
    from paper_1109_4279_gb300 import binding
    dims = (8, 8, 8, 16)
    U, rng = synth.gauge_field(dims, spread, 5)
    eta = synth.gaussian_spinor(dims, rng)
    A = orc.clover(dims, U, m0, 1.5)
    lat = binding.Lattice(dims, block, m0, 1.5)
    lat.load_gauge(torch.from_numpy(U).cuda())
    inside = np.zeros(dims, bool)
    inside[tuple(slice(b) for b in block)] = True
    inside = inside.reshape(-1)
    for nmr in (64, 128):
        psi = lat.sap(torch.from_numpy(eta).cuda(), ncy=1, nmr=nmr, prec=prec).cpu().numpy()
        assert np.isfinite(psi).all()
        psi[~inside] = 0
        r = (eta - orc.apply_D(dims, U, A, synth.ANTIPERIODIC_T, psi))[inside]
        assert np.linalg.norm(r) < TOL[prec] * np.linalg.norm(eta[inside])
    lat.close()

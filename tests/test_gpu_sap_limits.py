"""The largest Schwarz blocks of each precision: those whose fields fit in shared
memory are solved, by kernels compiled for no more threads than these blocks take, and
the next larger ones are refused before anything is launched.
"""
import pytest

from helpers import rel
from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

UNSUPPORTED = -11


@pytest.mark.parametrize("prec,block,fits", [
    ("f64", (2, 2, 6, 6), True), ("f64", (2, 2, 4, 10), False),      # 144 and 160 sites
    ("f32", (2, 4, 4, 10), True), ("f32", (2, 2, 6, 14), False),     # 320 and 336
    ("f16", (2, 4, 8, 8), True), ("f16", (2, 2, 10, 14), False),     # 512 and 560
], ids=str)
def test_largest_blocks(orc, prec, block, fits):
    from paper_1109_4279_gb300 import binding as B
    dims = tuple(2 * b for b in block)
    U, rng = synth.gauge_field(dims, 0.5, 44)
    eta = synth.gaussian_spinor(dims, rng)
    lat = B.Lattice(dims, block, 0.0, 1.2)
    lat.load_gauge(torch.from_numpy(U).cuda())
    et = torch.from_numpy(eta).cuda()
    psi = torch.empty_like(et)
    st = B.lib().qcd_sap_apply(lat.ctx, B._ptr(et), B._ptr(psi), 2, 4, B.PREC[prec], B._stream())
    lat.close()
    if not fits:
        assert st == UNSUPPORTED
        return
    assert st == 0
    ref = orc.sap(dims, U, orc.clover(dims, U, 0.0, 1.2), synth.ANTIPERIODIC_T, block, eta, 2, 4)
    assert rel(psi.cpu().numpy(), ref) < {"f64": 1e-12, "f32": 1e-5, "f16": 5e-3}[prec]

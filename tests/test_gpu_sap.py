"""The Schwarz preconditioner where its block solve can go wrong: no MR step
and an odd number of them, one cycle (nothing received) and several, blocks
with fewer pairs of sites than a warp and with extents that are no power of two,
right-hand sides one at a time and in tiles.
"""
import numpy as np
import pytest

from helpers import rel
from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5, "f16": 5e-3, "bf16": 4e-2}  # bf16: 8 bits of significand against f16's 11


@pytest.mark.parametrize("dims,block,precs", [
    ((4, 4, 4, 4), (2, 2, 2, 2), ("f64", "f32", "f16")),        # 8 pairs: most of a warp idle
    ((4, 8, 12, 4), (2, 4, 6, 2), ("f64", "f32", "f16")),       # 48 pairs
    ((12, 4, 4, 8), (6, 2, 2, 4), ("f32", "bf16")),
    ((8, 8, 8, 16), (4, 4, 4, 4), ("f32", "f16")),
    ((16, 8, 8, 8), (8, 4, 4, 4), ("f16", "bf16")),
], ids=str)
@pytest.mark.parametrize("ncy,nmr", [(1, 0), (1, 1), (2, 3), (3, 4)])
def test_sap(orc, dims, block, precs, ncy, nmr):
    from paper_1109_4279_gb300 import binding
    U, rng = synth.gauge_field(dims, 0.5, 91)
    eta = synth.gaussian_spinor(dims, rng, nrhs=3)
    A = orc.clover(dims, U, -0.05, 1.5)
    ref = [orc.sap(dims, U, A, synth.ANTIPERIODIC_T, block, e, ncy, nmr) for e in eta]
    lat = binding.Lattice(dims, block, -0.05, 1.5)
    lat.load_gauge(torch.from_numpy(U).cuda())
    et = torch.from_numpy(eta).cuda()
    for prec in precs:
        one = [lat.sap(et[k].contiguous(), ncy=ncy, nmr=nmr, prec=prec) for k in range(3)]
        for k in range(3):
            assert rel(one[k].cpu().numpy(), ref[k]) < TOL[prec]
        for rt in (1, 2, 3):  # tiles of right-hand sides: the same arithmetic
            psi = torch.empty_like(et)
            binding.qcd_sap_apply_n(lat.ctx, et, psi, 3, rt, ncy, nmr, prec)
            assert all(torch.equal(psi[k], one[k]) for k in range(3))
    lat.close()

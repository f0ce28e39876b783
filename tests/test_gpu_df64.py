"""The double-float operator over CTA sizes that leave the last CTA partly
empty, blocks of several shapes, and every boundary sign.
"""
import numpy as np
import pytest

from helpers import rel
from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,block,bc", [
    ((4, 4, 4, 4), (2, 2, 2, 2), (-1, 1, 1, 1)),
    ((4, 8, 12, 4), (2, 4, 6, 2), (1, -1, 1, -1)),
    ((8, 4, 4, 8), (4, 2, 2, 4), (-1, -1, -1, -1)),
    ((16, 8, 8, 8), (8, 4, 4, 4), (1, 1, -1, 1)),
], ids=str)
@pytest.mark.parametrize("dagger", [False, True])
def test_double_float_operator(orc, dims, block, bc, dagger):
    """Against the FP64 oracle: inputs split at 2^-49, products and sums rounded
    at about 2^-47 of their terms, 24 of them per result -- 2e-14 norm-wise;
    the CTA size changes nothing."""
    from paper_1109_4279_gb300 import binding
    U, rng = synth.gauge_field(dims, 0.5, 81)
    b = synth.gaussian_spinor(dims, rng, nrhs=2)
    lat = binding.Lattice(dims, block, -0.05, 1.5, bc)
    lat.load_gauge(torch.from_numpy(U).cuda())
    A = orc.clover(dims, U, -0.05, 1.5)
    bt = torch.from_numpy(b).cuda()
    out = lat.apply_D(bt, dagger=dagger, prec="df64")
    for k in range(2):
        assert rel(out[k].cpu().numpy(), orc.apply_D(dims, U, A, bc, b[k], dagger=dagger)) < 2e-14
    for threads in (32, 96, 160, 256):
        binding.qcd_set_launch(lat.ctx, "df64", threads, 1)
        assert torch.equal(lat.apply_D(bt, dagger=dagger, prec="df64"), out)
    lat.close()

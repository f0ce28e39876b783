"""The operator's launch shape: a size that the caller sets is the one that runs,
also where the FP64 operator would otherwise share a site among four warps.
"""
import pytest

from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,block", [((4, 4, 4, 4), (2, 2, 2, 2)), ((8, 8, 16, 16), (4, 4, 4, 4))], ids=str)
def test_fp64_size_that_was_set(orc, dims, block):
    """The two forms of the FP64 operator add the hops in different orders, and which
    one runs depends on the number of right-hand sides; with a size set, one right-hand
    side and several go through the same form and agree bit for bit."""
    from paper_1109_4279_gb300 import binding as B
    U, rng = synth.gauge_field(dims, 0.5, 81)
    psi = synth.gaussian_spinor(dims, rng, nrhs=3)
    ref = orc.apply_D(dims, U, orc.clover(dims, U, 0.1, 1.3), synth.ANTIPERIODIC_T, psi[0])
    lat = B.Lattice(dims, block, 0.1, 1.3)
    lat.load_gauge(torch.from_numpy(U).cuda())
    pt = torch.from_numpy(psi).cuda()
    default = lat.apply_D(pt, prec="f64")
    outs = []
    for threads in (32, 64, 512):
        B.qcd_set_launch(lat.ctx, "f64", threads)
        assert B.qcd_get_launch(lat.ctx, "f64") == (threads, 1)
        for n in (1, 2, 3):
            outs.append(lat.apply_D(pt[:n].contiguous(), prec="f64")[0])
    lat.close()
    assert all(torch.equal(o, outs[0]) for o in outs)
    for o in (default[0], outs[0]):
        assert abs(o.cpu().numpy() - ref).max() < 1e-13 * abs(ref).max()


def test_default_size(orc):
    """The default CTA size at the lattice sizes around which it changes (an SM's CTAs of
    128 and of 256 threads hold as many threads at the most from 19457 to 38912 and from
    58369 to 77824 sites on 152 SMs), and the operator with it."""
    import numpy as np
    from paper_1109_4279_gb300 import binding as B
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for dims, block in (((4, 4, 4, 4), (2, 2, 2, 2)), ((8, 8, 16, 16), (4, 4, 4, 4)), ((16, 12, 12, 12), (4, 6, 2, 2)),
                        ((8, 16, 16, 16), (4, 4, 4, 4)), ((24, 12, 12, 12), (4, 6, 2, 2)), ((16, 16, 16, 16), (4, 4, 4, 4)),
                        ((16, 16, 16, 20), (4, 4, 4, 2)), ((32, 16, 16, 16), (4, 4, 4, 4))):
        V = int(np.prod(dims))
        per_sm = [-(-(-(-V // t)) // sms) * t for t in (128, 256)]
        want = 256 if per_sm[1] <= per_sm[0] <= 512 else 128
        lat = B.Lattice(dims, block, 0.1, 1.3)
        assert [B.qcd_get_launch(lat.ctx, p) for p in ("f64", "f32", "f16", "bf16", "df64")] == [(want, 1)] * 4 + [(128, 1)]
        lat.close()

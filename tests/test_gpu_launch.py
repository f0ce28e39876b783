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


def test_autotune_keeps_the_default_within_reach(tmp_path):
    """The default sizes are among those that are timed; where the FP64 operator shares
    a site among four warps none is chosen for it, and it keeps doing so; a size set
    before the tuning no longer holds."""
    import json
    from paper_1109_4279_gb300 import binding as B
    for dims, block, small in (((8, 8, 8, 8), (4, 4, 4, 4), True), ((32, 16, 16, 16), (4, 4, 4, 4), False)):
        U, rng = synth.gauge_field(dims, 0.5, 82)
        U = torch.from_numpy(U).cuda()
        psi = torch.from_numpy(synth.gaussian_spinor(dims, rng)).cuda()
        lat = B.Lattice(dims, block, 0.1, 1.3)
        lat.load_gauge(U)
        default = B.qcd_get_launch(lat.ctx, "f64")
        assert default[0] in (128, 256, 512)
        want = lat.apply_D(psi, prec="f64")
        cache = tmp_path / ("tune%d.json" % lat.V)
        if small:
            B.qcd_set_launch(lat.ctx, "f64", 512)
            assert not torch.equal(lat.apply_D(psi, prec="f64"), want)
        B.qcd_autotune(lat.ctx, 1, str(cache))
        (key, vals), = json.load(open(cache)).items()
        assert B.qcd_get_launch(lat.ctx, "f64") == (vals[0], 1)
        if small:
            assert vals[0] == default[0] and torch.equal(lat.apply_D(psi, prec="f64"), want)
        lat.close()


def _write(cache, entries):
    """The cache's own layout: one entry per line."""
    cache.write_text("{\n" + ",\n".join('  "%s": %s' % (k, v) for k, v in entries.items()) + "\n}\n")


def test_cache_entries_of_other_kernels_are_not_applied(tmp_path):
    import json
    from paper_1109_4279_gb300 import binding as B
    dims, block = (8, 8, 8, 8), (4, 4, 4, 4)
    U, _ = synth.gauge_field(dims, 0.5, 83)
    lat = B.Lattice(dims, block, 0.1, 1.3)
    lat.load_gauge(torch.from_numpy(U).cuda())
    cache = tmp_path / "tune.json"
    B.qcd_autotune(lat.ctx, 1, str(cache))
    (key, vals), = json.load(open(cache)).items()
    unmarked = key[:key.index("|nrhs1") + len("|nrhs1")]
    assert unmarked != key
    old = [512, 512, 512, 512, 256, 2, 2, 0]
    _write(cache, {unmarked: old})
    B.qcd_set_launch(lat.ctx, "f64", 1024)
    B.qcd_autotune(lat.ctx, 1, str(cache))
    entries = json.load(open(cache))
    assert set(entries) == {unmarked, key} and entries[unmarked] == old
    assert B.qcd_get_launch(lat.ctx, "f64")[0] == entries[key][0] != 512
    entries[key] = old  # an entry of these kernels is applied as it stands
    _write(cache, entries)
    B.qcd_autotune(lat.ctx, 1, str(cache))
    assert B.qcd_get_launch(lat.ctx, "f32") == (512, 1) and B.qcd_get_launch(lat.ctx, "f16") == (256, 2)
    lat.close()

"""GPU fermion force where its kernels can go wrong: blocks and extents that
are no power of two, sites that do not fill the last CTA, no clover term, and
lattices so large that the planes are taken one at a time.
"""
import numpy as np
import pytest

from helpers import vdot
from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

AP = synth.ANTIPERIODIC_T


@pytest.mark.parametrize("dims,block,csw", [
    ((4, 4, 4, 4), (2, 2, 2, 2), 1.3),
    ((4, 8, 12, 4), (2, 4, 6, 2), 1.2),   # 1536 sites, blocks of 96
    ((12, 4, 4, 20), (6, 2, 2, 2), 0.7),  # 3840 sites, blocks of 48
    ((8, 4, 4, 8), (4, 2, 2, 4), 0.0),    # hopping part alone
], ids=str)
def test_force_along_random_directions(orc, dims, block, csw):
    """theta . F = -Re(y^+ dD x) with the oracle's dD for directions theta over
    all links: rounding of N = 32 V terms stays below 1e-13 |theta| |F|."""
    from paper_1109_4279_gb300 import binding
    U, rng = synth.gauge_field(dims, 0.5, 62)
    x, y = synth.gaussian_spinor(dims, rng), synth.gaussian_spinor(dims, rng)
    lat = binding.Lattice(dims, block, 0.1, csw)
    lat.load_gauge(torch.from_numpy(U).cuda())
    F = torch.empty((lat.V, 4, 8), dtype=torch.float64, device="cuda")
    binding.qcd_force(lat.ctx, torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), F)
    F = F.cpu().numpy()
    for k in range(8):
        theta = rng.standard_normal((lat.V, 4, 8))
        if k >= 4:  # one direction alone
            theta *= (np.arange(4) == k - 4)[None, :, None]
        d = orc.dD_apply(dims, U, 1j * np.einsum("vmab,vmbc->vmac", synth.algebra(theta), U), AP, csw, x)
        assert abs(np.sum(theta * F) + np.real(vdot(y, d))) < 1e-13 * np.linalg.norm(theta) * np.linalg.norm(F)
    lat.close()


def test_force_plane_by_plane_equals_all_planes():
    """A lattice made of two copies of a smaller one side by side (periodic, so
    the force of either half is the smaller one's): the smaller takes its six
    planes in one launch, the larger (over 4 GiB for six) one by one.  Same
    arithmetic in the same order: equal bit for bit."""
    from paper_1109_4279_gb300 import binding
    small, large = (48, 32, 32, 24), (48, 32, 32, 48)
    assert 6 * 41 * 8 * np.prod(small) <= 4 << 30 < 6 * 41 * 8 * np.prod(large)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    V = int(np.prod(small))
    U = torch.eye(3, dtype=torch.complex128, device="cuda").expand(V, 4, 3, 3).contiguous()
    pi = torch.randn((V, 4, 8), dtype=torch.float64, device="cuda", generator=gen)
    x, y = (torch.view_as_complex(torch.randn((V, 4, 3, 2), dtype=torch.float64, device="cuda", generator=gen))
            for _ in range(2))

    def twice(t):
        t = t.reshape(*small, *t.shape[1:])
        return torch.cat((t, t), dim=3).reshape(-1, *t.shape[4:]).contiguous()

    out = []
    for dims, dup in ((small, lambda t: t), (large, twice)):
        lat = binding.Lattice(dims, (4, 4, 4, 4), 0.1, 1.5)
        if dup is not twice:
            binding.qcd_update_links(lat.ctx, U, pi, 0.5)
        lat.load_gauge(dup(U))
        F = torch.empty((lat.V, 4, 8), dtype=torch.float64, device="cuda")
        binding.qcd_force(lat.ctx, dup(x), dup(y), F)
        out.append(F)
        lat.close()
    assert torch.equal(twice(out[0]), out[1])

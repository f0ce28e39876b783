"""Forces and momenta in arrays that start at an odd element of a larger one
(8-byte aligned, not 16): the results are those of an array of their own, bit for
bit, and the elements around them stay as they are.
"""
import pytest

from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GUARD = 7.25


def _offset(values):
    """The values one element into an allocation of their own, guards on both sides
    (the view is only passed on, never computed with)."""
    host = torch.full((len(values) + 3,), GUARD, dtype=torch.float64)
    host[1:-2] = values
    buf = host.cuda()
    view = buf[1:-2]
    assert view.data_ptr() % 16 == 8 and view.is_contiguous()
    return buf, view


def _check(buf, want):
    got = buf.cpu()
    assert torch.equal(got[1:-2], want.cpu().reshape(-1))
    assert got[0] == GUARD and bool((got[-2:] == GUARD).all())


@pytest.mark.parametrize("dims,block", [
    ((8, 4, 4, 4), (2, 2, 2, 2)),
    ((12, 4, 4, 64), (2, 2, 2, 4)),  # 12288 sites: the gauge force goes by plaquettes
], ids=str)
def test_force_and_momenta(dims, block):
    from paper_1109_4279_gb300 import binding as B
    U, rng = synth.gauge_field(dims, 0.5, 41)
    U = torch.from_numpy(U).cuda()
    x, y = (torch.from_numpy(synth.gaussian_spinor(dims, rng)).cuda() for _ in range(2))
    lat = B.Lattice(dims, block, 0.1, 1.2)
    lat.load_gauge(U)
    n = lat.V * 32
    empty = torch.zeros(n, dtype=torch.float64)
    own = torch.empty(n, dtype=torch.float64, device="cuda")
    sp = B.solver_params(tol=1e-8)
    for call in (lambda F: B.qcd_force(lat.ctx, x, y, F), lambda F: B.qcd_gauge_force(lat.ctx, U, 5.4, F),
                 lambda F: B.qcd_gradient(lat.ctx, x, dL_dtheta=F, params=sp)):
        buf, F = _offset(empty)
        call(own)
        call(F)
        torch.cuda.synchronize()
        _check(buf, own)

    momenta = torch.from_numpy(rng.standard_normal(n))
    buf, pi = _offset(momenta)
    A, C = U.clone(), U.clone()
    B.qcd_update_links(lat.ctx, A, momenta.cuda(), 0.3)
    B.qcd_update_links(lat.ctx, C, pi, 0.3)
    assert torch.equal(A, C)
    _check(buf, momenta)
    lat.close()


def test_trajectory_momenta():
    from paper_1109_4279_gb300 import binding as B
    dims, block = (4, 4, 4, 8), (2, 2, 2, 2)
    U, rng = synth.gauge_field(dims, 0.3, 42)
    U = torch.from_numpy(U).cuda()
    eta = torch.from_numpy(synth.gaussian_spinor(dims, rng)).cuda()
    lat = B.Lattice(dims, block, 0.3, 1.0)
    momenta = torch.from_numpy(rng.standard_normal(lat.V * 32))
    buf, pi = _offset(momenta)
    own = momenta.cuda()
    sp = B.solver_params(tol=1e-10)
    A, C = U.clone(), U.clone()
    a = B.qcd_hmc_trajectory(lat.ctx, A, own, eta, 5.4, 0.05, 2, 0.0, sp)
    c = B.qcd_hmc_trajectory(lat.ctx, C, pi, eta, 5.4, 0.05, 2, 0.0, sp)
    assert a["dH"] == c["dH"] and torch.equal(A, C)
    _check(buf, own)
    lat.close()

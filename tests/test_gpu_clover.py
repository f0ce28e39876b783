"""GPU clover build: the leaves' exchange between sites and the inverse of the
chiral blocks, on smooth links (every pivot on the diagonal) and on random ones
with a small mass, where many blocks need pivoting.
"""
import numpy as np
import pytest

from helpers import rel
from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

AP = synth.ANTIPERIODIC_T


def _lexicographic(dims):
    return np.stack(np.meshgrid(*(np.arange(d) for d in dims), indexing="ij"), -1).reshape(-1, 4)


@pytest.mark.parametrize("dims,block,links,m0,csw", [
    ((4, 4, 4, 4), (2, 2, 2, 2), "smooth", 0.1, 1.0),
    ((4, 8, 12, 4), (2, 4, 6, 2), "smooth", -0.05, 1.5),   # 1536 sites, blocks of 96
    ((12, 4, 4, 20), (6, 2, 2, 2), "smooth", 0.0, 0.0),    # no clover term
    ((4, 8, 12, 4), (2, 4, 6, 2), "random", -3.7, 1.9),
], ids=str)
def test_clover_and_its_inverse(orc, dims, block, links, m0, csw):
    """D psi gives A; one SAP half-sweep of no MR steps leaves psi_o = A_oo^-1 eta_o
    on the odd sites of the blocks solved first.  Both against the oracle's A: A to
    1e-13, the inverse to 1e-14 times each site's condition number."""
    from paper_1109_4279_gb300 import binding
    rng = np.random.default_rng(17)
    V = int(np.prod(dims))
    U = synth.gauge_field(dims, 0.5, 17, rng=rng)[0] if links == "smooth" else \
        synth.random_su3(4 * V, rng).reshape(V, 4, 3, 3)
    eta = synth.gaussian_spinor(dims, rng)
    lat = binding.Lattice(dims, block, m0, csw)
    lat.load_gauge(torch.from_numpy(U).cuda())
    A = orc.clover(dims, U, m0, csw)
    et = torch.from_numpy(eta).cuda()
    assert rel(lat.apply_D(et).cpu().numpy(), orc.apply_D(dims, U, A, AP, eta)) < 1e-13
    psi = lat.sap(et, ncy=1, nmr=0, prec="f64").cpu().numpy().reshape(V, 12)
    x = _lexicographic(dims)
    pick = (x.sum(1) % 2 == 1) & ((x // np.array(block)).sum(1) % 2 == 0)
    ref = np.linalg.solve(A[pick], eta.reshape(V, 12)[pick][..., None])[..., 0]
    cond = np.linalg.cond(A[pick])
    off = np.linalg.norm(psi[pick] - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert np.all(off < 1e-14 * cond)
    lead = np.abs(A[pick][:, 1:6, 0].real) + np.abs(A[pick][:, 1:6, 0].imag)
    assert np.any(lead.max(1) > np.abs(A[pick][:, 0, 0])) == (links == "random")
    lat.close()


def test_singular_clover_is_refused_and_the_context_recovers(orc):
    """m0 = -4 without clover term: every block is 0.  The next build on the
    same context (whose records are kept) after a good one gives D again."""
    from paper_1109_4279_gb300 import binding
    dims, block = (4, 4, 4, 4), (2, 2, 2, 2)
    U, rng = synth.gauge_field(dims, 0.3, 3)
    lat = binding.Lattice(dims, block, -4.0, 0.0)
    binding.qcd_load_gauge(lat.ctx, torch.from_numpy(U).cuda())
    with pytest.raises(binding.QcdError, match="QCD_ERR_SINGULAR_CLOVER"):
        binding.qcd_build_clover(lat.ctx)
    with pytest.raises(binding.QcdError, match="QCD_ERR_STATE"):
        lat.apply_D(torch.from_numpy(synth.gaussian_spinor(dims, rng)).cuda())
    lat.close()
    lat = binding.Lattice(dims, block, 0.1, 1.0)
    psi = synth.gaussian_spinor(dims, rng)
    for seed in (3, 4):  # a second field on the same context
        U, _ = synth.gauge_field(dims, 0.3, seed)
        lat.load_gauge(torch.from_numpy(U).cuda())
        out = lat.apply_D(torch.from_numpy(psi).cuda(), prec="df64").cpu().numpy()
        assert rel(out, orc.apply_D(dims, U, orc.clover(dims, U, 0.1, 1.0), AP, psi)) < 1e-12
    lat.close()

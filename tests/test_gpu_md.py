"""The gauge half of molecular dynamics at the edges of its kernels: every
branch of the link exponential.
"""
import numpy as np
import pytest

from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [0.0, 1e-9, 0.02, 0.1, 0.4, 0.9, 3.0, 50.0])
def test_link_update(eps):
    """exp(i eps P) U over all links against the eigen-decomposition, momenta of
    every size among them: the series' lengths (|H| to 0.06, 1/4, 1, 2) and the
    squarings beyond.  Rounding grows with |H|: 1e-14 (1 + |H|)."""
    from paper_1109_4279_gb300 import binding
    dims = (4, 4, 4, 12)  # 3072 links
    U, rng = synth.gauge_field(dims, 0.5, 71)
    pi = rng.standard_normal((U.shape[0], 4, 8)) * 10.0 ** rng.uniform(-2, 0.5, (U.shape[0], 4, 1))
    pi[0, 0] = 0.0
    pi[0, 1] = [0, 0, 1, 0, 0, 0, 0, 1]  # diagonal P
    lat = binding.Lattice(dims, (2, 2, 2, 2), 0.0, 0.0)
    Ut = torch.from_numpy(U).cuda()
    binding.qcd_update_links(lat.ctx, Ut, torch.from_numpy(pi).cuda(), eps)
    H = eps * synth.algebra(pi)
    w, v = np.linalg.eigh(H)
    E = np.einsum("...ab,...b,...cb->...ac", v, np.exp(1j * w), np.conj(v))
    off = np.abs(Ut.cpu().numpy() - np.einsum("...ab,...bc->...ac", E, U)).max(axis=(2, 3))
    assert np.all(off < 1e-14 * (1 + np.linalg.norm(H, axis=(2, 3))))
    lat.close()

"""The gauge half of molecular dynamics at the edges of its kernels: every
branch of the link exponential, and the gauge force on both sides of the size
from which it goes by plaquettes.
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


@pytest.mark.parametrize("dims", [
    (4, 4, 4, 4),
    (4, 12, 4, 20),   # 3840 sites, one thread per link
    (12, 4, 4, 64),   # 12288 sites, the smallest that goes by plaquettes
    (28, 4, 20, 8),   # 17920 sites: a last CTA of half its threads in every round
    (4, 36, 12, 8),
], ids=str)
def test_gauge_force(dims):
    """F = dS/dtheta of the plaquette action by torch's derivative in FP64 on the
    CPU; sums of six staples: 1e-13 of the field's norm."""
    from paper_1109_4279_gb300 import binding
    U, _ = synth.gauge_field(dims, 0.7, 72)
    lat = binding.Lattice(dims, (2, 2, 2, 2), 0.0, 0.0)
    F = torch.full((lat.V, 4, 8), float("nan"), dtype=torch.float64, device="cuda")
    binding.qcd_gauge_force(lat.ctx, torch.from_numpy(U).cuda(), 5.3, F)
    theta = torch.zeros((lat.V, 4, 8), dtype=torch.float64, requires_grad=True)
    lam = torch.from_numpy(synth.GELL_MANN) / 2
    u = torch.from_numpy(U)
    w = (u + 1j * torch.einsum("vma,aij->vmij", theta.to(torch.complex128), lam) @ u).reshape(*dims, 4, 3, 3)
    S = 0.0
    for m in range(4):
        for n in range(m + 1, 4):
            a, b = w[..., m, :, :], w[..., n, :, :]
            P = a @ torch.roll(b, -1, dims=m) @ torch.roll(a, -1, dims=n).mH @ b.mH
            S = S + 5.3 * (1.0 - torch.einsum("...ii->...", P).real / 3.0).sum()
    ref = torch.autograd.grad(S, theta)[0]
    assert torch.linalg.vector_norm(F.cpu() - ref) < 1e-13 * torch.linalg.vector_norm(ref)
    lat.close()

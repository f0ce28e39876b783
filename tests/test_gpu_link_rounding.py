"""The rounding of the link update's exponential, against extended precision: links
of 1, so that exp(i H) itself comes back, for random H and for H with two (nearly)
equal eigenvalues, small steps and steps far beyond a molecular-dynamics one.
"""
import numpy as np
import pytest

from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U_ROUND = 2.0 ** -53


def _mm(a, b):
    return np.einsum("...ij,...jk->...ik", a, b)


def _exp_i(H):
    """exp(i H) in numpy's extended precision: 20 Taylor terms of H / 2^k, |H / 2^k| < 1/8."""
    k = max(0, int(np.ceil(np.log2(float(np.sqrt((np.abs(H) ** 2).sum((-1, -2))).max())))) + 3)
    A = 1j * H / np.longdouble(2) ** k
    one = np.eye(3, dtype=np.clongdouble)
    E = np.broadcast_to(one, A.shape)
    for m in range(20, 0, -1):
        E = one + _mm(A, E) / np.longdouble(m)
    for _ in range(k):
        E = _mm(E, E)
    return E


def _momenta(n, kind, rng):
    if kind == "random":
        return rng.standard_normal((n, 8))
    # eigenvalues 1 + g, 1 - g, -2 (or their negatives) in random bases
    q, _ = np.linalg.qr(rng.standard_normal((n, 3, 3)) + 1j * rng.standard_normal((n, 3, 3)))
    g = 10.0 ** rng.uniform(-16, -1, n) * (rng.random(n) > 0.3)
    w = np.stack([1 + g, 1 - g, np.full(n, -2.0)], -1) * rng.choice([-1.0, 1.0], (n, 1))
    H = np.einsum("nij,nj,nkj->nik", q, w, q.conj())
    return np.einsum("aij,nji->na", synth.GELL_MANN, H).real


@pytest.mark.parametrize("size", [0.01, 0.05, 0.2, 0.9, 1.9, 2.1, 6.0, 32.0, 100.0, 1e3, 1e5])
def test_exponential(size):
    """Up to |H| = 1/4 every real of exp(i H) is rounded once after a correction of
    at most |H|: one unit u.  Beyond, a relative error of 8 u in H and in each squaring's
    result, which the squarings pass on as 8 u |H|."""
    from paper_1109_4279_gb300 import binding
    dims = (4, 4, 4, 8)  # 2048 links
    rng = np.random.default_rng(17)
    V = int(np.prod(dims))
    pi = np.concatenate([_momenta(2 * V, k, rng) for k in ("random", "degenerate")])
    pi *= size / np.sqrt(0.5 * (pi ** 2).sum(-1, keepdims=True))  # |H|^2 = sum pi^2 / 2
    lam = synth.GELL_MANN.astype(np.clongdouble)
    lam[7] *= 1 / (np.sqrt(np.longdouble(3)) * lam[7][0, 0])  # (1/sqrt 3 in extended precision)
    H = np.einsum("na,aij->nij", pi.astype(np.longdouble), lam) / 2
    U = torch.eye(3, dtype=torch.complex128, device="cuda").expand(V, 4, 3, 3).contiguous()
    lat = binding.Lattice(dims, (2, 2, 2, 2), 0.0, 0.0)
    binding.qcd_update_links(lat.ctx, U, torch.from_numpy(pi).cuda(), 1.0)
    lat.close()
    d = U.cpu().numpy().reshape(-1, 3, 3) - _exp_i(H)
    off = float(max(np.abs(d.real).max(), np.abs(d.imag).max()))
    assert off < (U_ROUND if size <= 0.25 else 8 * U_ROUND * max(1.0, size))

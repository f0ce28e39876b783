"""The Krylov recursion's vector kernels over every number of basis vectors
they have an instance for: unpreconditioned solves need more iterations than
the restart length, so k runs through 0 .. nkv - 1.
"""
import numpy as np
import pytest

from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

AP = synth.ANTIPERIODIC_T


@pytest.mark.parametrize("dims,block", [((4, 4, 4, 4), (2, 2, 2, 2)), ((4, 8, 12, 4), (2, 4, 6, 2))], ids=str)
@pytest.mark.parametrize("outer", ["df64", "f64", "f32"])
@pytest.mark.parametrize("nkv,nrhs", [(1, 1), (3, 1), (9, 2), (20, 1), (33, 1)])
def test_unpreconditioned_restarts(orc, dims, block, outer, nkv, nrhs):
    """GCR(nkv) to 1e-10 on a well-conditioned operator: the true residual is the
    oracle's, and the recursions in double-float and FP64 take the same number of
    iterations (FP32 cycles end early by design)."""
    from paper_1109_4279_gb300 import binding
    U, rng = synth.gauge_field(dims, 0.3, 51)
    b = synth.gaussian_spinor(dims, rng, nrhs=nrhs)
    lat = binding.Lattice(dims, block, 0.5, 1.0)
    lat.load_gauge(torch.from_numpy(U).cuda())
    bt = torch.from_numpy(b).cuda()
    x, info = lat.solve(bt, tol=1e-10, precond="none", outer_prec=outer, nkv=nkv, max_restarts=400)
    assert any(i["iterations"] > nkv for i in info)
    A = orc.clover(dims, U, 0.5, 1.0)
    for k in range(nrhs):
        r = b[k] - orc.apply_D(dims, U, A, AP, x[k].cpu().numpy())
        assert np.linalg.norm(r) <= 1.01e-10 * np.linalg.norm(b[k])
    if outer == "df64":
        _, ref = lat.solve(bt, tol=1e-10, precond="none", outer_prec="f64", nkv=nkv, max_restarts=400)
        assert [i["iterations"] for i in ref] == [i["iterations"] for i in info]
    lat.close()

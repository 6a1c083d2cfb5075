"""Restart lengths of the interface GMRES near the longest that is taken (1599):
the solution of the default length, and longer ones are refused.

Both solves end at a relative residual of 1e-10; cond of the global matrix is
below 1e4 at this size: 1e-6."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("restart", [1536, 1537, 1599])
def test_long_outer_restart(restart):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2105_11993_gb300 as thm
    P = W.square_problem(12, 2, 1, 9.0, mu_inv=W.mu_inv_lognormal(144, 0.3, "outer"))
    mesh = thm.Mesh.from_workload(P.mesh, P.order)
    s = thm.System(mesh, P.mu_inv, P.omega, P.kappa, P.pol, P.direction)
    a, st = s.solve(mode="fp64", rtol=1e-10, outer_restart=restart)
    s = thm.System(mesh, P.mu_inv, P.omega, P.kappa, P.pol, P.direction)
    b, _ = s.solve(mode="fp64", rtol=1e-10)
    assert float((a - b).norm() / b.norm()) <= 1e-6
    with pytest.raises(thm.ThmError) as e:
        thm.System(mesh, P.mu_inv, P.omega, P.kappa, P.pol, P.direction).solve(mode="fp64", outer_restart=1600)
    assert e.value.code == -1

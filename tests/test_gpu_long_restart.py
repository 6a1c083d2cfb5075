"""Restart lengths near the largest that is taken (FP64 1599, mixed 799): the
scalars of such cycles outgrow shared memory, and the solve still gives the
sweep of the default length; longer ones are refused.

Both stop at a residual of 1e-13 and cond(T_i) is below 1e4 here: 1e-9."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("mode,longest", [("fp64", 1599), ("mixed", 799)])
def test_longest_restart(mode, longest):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2105_11993_gb300 as thm
    P = W.square_problem(12, 2, 2, 9.0, mu_inv=W.mu_inv_lognormal(144, 0.3, "sweep"))
    mesh = thm.Mesh.from_workload(P.mesh, P.order)
    outs = []
    for m in (longest, 0):
        s = thm.System(mesh, P.mu_inv, P.omega, P.kappa, P.pol, P.direction)
        g = 1e-2 * torch.randn(s.n_iface, dtype=torch.complex128, device="cuda",
                               generator=torch.Generator("cuda").manual_seed(1))
        outs.append(s.sweep(g, mode=mode, inner_tol=1e-13, inner_restart=m)[:2])
    for a, b in zip(*outs):
        assert float((a - b).norm() / b.norm()) <= 1e-9
    with pytest.raises(thm.ThmError):
        s = thm.System(mesh, P.mu_inv, P.omega, P.kappa, P.pol, P.direction)
        s.sweep(g, mode=mode, inner_restart=longest + 1)

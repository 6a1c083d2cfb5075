"""A sweep as the first call on a system builds the factors of the
preconditioner that its options name (the full 2x2 block operator's complex
factors too), so it gives the same sweep as with the default preconditioner."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("mode", ["fp64", "mixed"])
def test_first_sweep_with_the_full_preconditioner(mode):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2105_11993_gb300 as thm
    P = W.square_problem(12, 2, 2, 9.0, mu_inv=W.mu_inv_lognormal(144, 0.3, "sweep"))
    mesh = thm.Mesh.from_workload(P.mesh, P.order)
    outs = []
    for precond in ("full", "blockdiag"):
        s = thm.System(mesh, P.mu_inv, P.omega, P.kappa, P.pol, P.direction)
        g = 1e-2 * torch.randn(s.n_iface, dtype=torch.complex128, device="cuda",
                               generator=torch.Generator("cuda").manual_seed(1))
        outs.append(s.sweep(g, mode=mode, inner_tol=1e-13, precond=precond)[:2])
    # both stop at a residual of 1e-13; cond(T_i) is below 1e4 here
    for a, b in zip(*outs):
        assert float((a - b).norm() / b.norm()) <= 1e-9

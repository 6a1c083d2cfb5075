"""Subdomain solves with the apply's vectors, its slice table and the Krylov
vectors in global memory (the form of subdomains that outgrow shared memory),
forced on ordinary sizes: one to eight CTAs per subdomain, both dimensions and
orders, both preconditioners.

The arithmetic and its order are the same, so the results agree to the rounding
that another contraction of multiply-adds may leave, amplified by the solve: both
end at a residual of 1e-12 and cond(T_i) is below 1e4: 1e-8."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2105_11993_gb300 import build
    build.build()


CASES = {
    "p2": lambda: W.square_problem(24, 2, 2, 9.0, mu_inv=W.mu_inv_lognormal(576, 0.3, "glob")),
    "p1_many": lambda: W.square_problem(60, 20, 1, 9.0, mu_inv=W.mu_inv_lognormal(3600, 0.3, "glob")),
    "near_resonance": lambda: W.square_problem(64, 2, 2, 25.132741228718345),
    "cube": lambda: W.cube_problem(8, 2, 6.0, mu_inv=W.mu_inv_lognormal(512, 0.3, "glob")),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("mode", ["fp64", "mixed"])
def test_sweep(name, mode, monkeypatch):
    import paper_2105_11993_gb300 as thm
    P = CASES[name]()
    s = thm.System(thm.Mesh.from_workload(P.mesh, P.order), P.mu_inv, P.omega, P.kappa, P.pol, P.direction)
    g = 1e-2 * torch.randn(s.n_iface, dtype=torch.complex128, device="cuda",
                           generator=torch.Generator("cuda").manual_seed(1))
    for precond in ["blockdiag"] + (["full"] if P.mesh.dim == 2 else []):
        a = s.sweep(g, mode=mode, inner_tol=1e-12, precond=precond)
        monkeypatch.setenv("THM_BT_CPL_GLOBAL", "1")
        b = s.sweep(g, mode=mode, inner_tol=1e-12, precond=precond)
        monkeypatch.delenv("THM_BT_CPL_GLOBAL")
        for x, y in zip(a[:2], b[:2]):
            assert float((x - y).norm() / x.norm()) <= 1e-8, precond

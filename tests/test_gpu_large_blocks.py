"""Nodes whose block outgrows shared memory in the factorisation: inverted a
panel of columns at a time, 16 or 8 wide by the size of the block, for real and
complex factors, at block sizes that are no multiple of a panel.

One subdomain each: the root, which joins the top three cuts, is the large node.
kappa = 0, so T_i P_i^{-1} x = x; tolerance as for the small trees (u cond(P_i)
times the growth of the elimination: 1e-8)."""
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
    "p1": lambda: (W.structured_mesh_2d(61, 67, 1, 1), 1),
    "p2": lambda: (W.structured_mesh_2d(43, 41, 1, 1), 2),
    "p2_wide": lambda: (W.structured_mesh_2d(110, 107, 1, 1), 2),       # panels of 8 complex columns
    "cube8": lambda: (W.structured_mesh_3d(8, 1), 1),
    "cube15": lambda: (W.structured_mesh_3d(15, 1), 1),
    "cube18": lambda: (W.structured_mesh_3d(18, 1), 1),                 # panels of 8 real columns
}


@pytest.mark.parametrize("name", list(CASES))
def test_operator_times_inverse_is_the_identity(name):
    import paper_2105_11993_gb300 as thm
    mesh, order = CASES[name]()
    mu = W.mu_inv_lognormal(mesh.n_cell, 0.3, "blocks/" + name)
    pol, d = W.plane_wave_y(mesh.dim)
    s = thm.System(thm.Mesh.from_workload(mesh, order), mu, 2.3, 0.0, pol, d)
    x = torch.randn(s.n_local, dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    for op in [thm.OP_PINV] + ([thm.OP_TINV] if mesh.dim == 2 else []):
        y = s.apply_local(op, x, mode="fp64")
        assert float((s.apply_local(thm.OP_T, y, mode="fp64") - x).norm() / x.norm()) <= 1e-8

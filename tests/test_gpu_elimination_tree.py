"""The nested-dissection factorisation and solve at the sizes where their
tables change shape: single cells, leaves that hold the whole subdomain, ragged
and lopsided subdomains, one to eight CTAs per subdomain (few large to many
small subdomains), and vectors that outgrow shared memory.

With kappa = 0 the subdomain operator T_i is P_i itself, so T_i P_i^{-1} x = x
without an oracle.  Tolerances: the elimination is backward stable up to the
growth of its Schur complements, so the residual is about u cond(P_i) times
that growth; at these frequencies cond <= 1e5 and growth <= 1e3, which gives
1e-16 * 1e8 = 1e-8 for FP64 factors.  FP32 factors (u = 6e-8) allow no such
bound beyond telling a wrong table (errors of order 1) from rounding:
cond * u = 6e-3 at cond 1e5, taken as 5e-2."""
import numpy as np
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


def _mesh_2d(nx, ny, sx, sy):
    return W.structured_mesh_2d(nx, ny, sx, sy, bc="impedance", relabel=True, rotate_cells=True)


CASES = {
    "one_cell": lambda: (_mesh_2d(1, 1, 1, 1), 1),
    "one_cell_p2": lambda: (_mesh_2d(1, 1, 1, 1), 2),
    "leaf": lambda: (_mesh_2d(4, 2, 1, 1), 1),
    "leaf_p2": lambda: (_mesh_2d(3, 1, 1, 1), 2),
    "strip": lambda: (_mesh_2d(37, 2, 2, 1), 2),
    "odd": lambda: (_mesh_2d(23, 17, 1, 1), 2),
    "odd_p1": lambda: (_mesh_2d(31, 29, 2, 3), 1),
    "c4": lambda: (_mesh_2d(64, 64, 8, 8), 1),
    "c2": lambda: (_mesh_2d(70, 70, 10, 10), 2),
    "c1": lambda: (_mesh_2d(80, 80, 20, 20), 1),
    "outgrows_smem": lambda: (_mesh_2d(96, 96, 1, 1), 2),
    "cube_cell": lambda: (W.structured_mesh_3d(1, 1, bc="planewave"), 1),
    "cube": lambda: (W.structured_mesh_3d(9, 1, relabel=True, rotate_cells=True), 1),
    "cube_many": lambda: (W.structured_mesh_3d(14, 7), 1),
}


def _system(name):
    import paper_2105_11993_gb300 as thm
    mesh, order = CASES[name]()
    mu = W.mu_inv_lognormal(mesh.n_cell, 0.3, "tree/" + name)
    pol, d = W.plane_wave_y(mesh.dim)
    m = thm.Mesh.from_workload(mesh, order)
    return thm, thm.System(m, mu, 2.3, 0.0, pol, d)


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("mode", ["fp64", "mixed"])
def test_operator_times_inverse_is_the_identity(name, mode):
    thm, s = _system(name)
    x = torch.randn(s.n_local, dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    y = s.apply_local(thm.OP_PINV, x, mode=mode)
    r = s.apply_local(thm.OP_T, y, mode="fp64") - x
    assert float(r.norm() / x.norm()) <= (1e-8 if mode == "fp64" else 5e-2)
    # a second apply gives the same bits: every sum has a fixed order
    assert torch.equal(y, s.apply_local(thm.OP_PINV, x, mode=mode))


@pytest.mark.parametrize("name", ["one_cell_p2", "odd", "odd_p1", "c2"])
def test_complex_factors_without_impedance_equal_the_real_ones(name):
    """B = 0 (kappa = 0): T_i^{-1} from complex factors is P_i^{-1}."""
    thm, s = _system(name)
    x = torch.randn(s.n_local, dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    y = s.apply_local(thm.OP_PINV, x, mode="fp64")
    z = s.apply_local(thm.OP_TINV, x, mode="fp64")
    assert float((y - z).norm() / y.norm()) <= 1e-8

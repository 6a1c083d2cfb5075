"""A subdomain whose P_i is exactly singular is THM_ESINGULAR also where other
subdomains of the system move unknowns up their trees (a uniform medium at 3.63
cells per wavelength does, in 2x2-cell cavities).

The singular one is a single square cell of side 1/32 whose permittivity
vanishes beside its curl term: P_i = 1024 (+-1) is of rank one, and every step
of the elimination is exact in binary."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _system(eps_of_cell):
    import paper_2105_11993_gb300 as thm
    mesh = W.structured_mesh_2d(49, 48)
    at = np.rint(mesh.coords * [49, 48]).astype(int)
    cell = at[mesh.cells].min(1)
    mesh.coords = at / 32.0
    mesh.cell_sub = (cell[:, 0] // 24 + 2 * (cell[:, 1] // 24)).astype(np.int32)
    mesh.cell_sub[cell[:, 0] == 48] = 5
    lone = (cell[:, 0] == 48) & (cell[:, 1] == 20)
    mesh.cell_sub[lone] = 4
    eps = np.ones(mesh.n_cell)
    eps[lone] = eps_of_cell
    pol, d = W.plane_wave_y(2)
    m = thm.Mesh.from_workload(mesh, 1)
    return thm, thm.System(m, np.ones(mesh.n_cell), 32 * 2 * np.pi / 3.6276, 0.0, pol, d, eps=eps)


@pytest.mark.parametrize("op", ["PINV", "TINV"])
def test_singular_beside_moves(op):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    thm, s = _system(1e-300)
    x = torch.randn(s.n_local, dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    with pytest.raises(thm.ThmError) as e:
        s.apply_local(getattr(thm, "OP_" + op), x, mode="fp64")
    assert e.value.code == -4
    # the same system with the cell as it was: P_i P_i^{-1} x = x (kappa = 0)
    thm, s = _system(1.0)
    y = s.apply_local(getattr(thm, "OP_" + op), x, mode="fp64")
    assert float((s.apply_local(thm.OP_T, y, mode="fp64") - x).norm() / x.norm()) <= 1e-8

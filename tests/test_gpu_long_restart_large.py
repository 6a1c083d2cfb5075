"""A mixed subdomain solve whose restart length leaves no shared memory for the
vectors of the preconditioner apply: one subdomain of 206x203 order-1 cells
(83,842 unknowns, 32-bit columns, odd lengths of the u buffers), u and the
staged y in the workspace.

The same sweep as at the default restart length: both stop at a residual of
1e-10 and cond(T_i) is below 1e4, so the solutions agree to 1e-6."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_vectors_in_the_workspace():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2105_11993_gb300 as thm
    mesh = W.structured_mesh_2d(206, 203, 1, 1)
    pol, d = W.plane_wave_y(2)
    s = thm.System(thm.Mesh.from_workload(mesh, 1), W.mu_inv_lognormal(mesh.n_cell, 0.3, "large"), 9.0, 1.0, pol, d)
    outs = []
    for m in (799, 0):
        g = torch.zeros(1, dtype=torch.complex128, device="cuda")
        outs.append(s.sweep(g, mode="mixed", inner_tol=1e-10, inner_restart=m)[1])
    assert float((outs[0] - outs[1]).norm() / outs[1].norm()) <= 1e-6

"""The interface GMRES on interfaces of fewer unknowns than one chunk holds, of
a few chunks, and of so many that a chunk is walked in several pieces (more than
152 * 128): the solve reaches its tolerance, measured by the FP64 true residual
that other kernels form."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,s,least,most", [(6, 2, 1, 128), (24, 3, 128, 1024), (160, 40, 152 * 128 + 1, 10 ** 6)])
def test_interface_sizes(n, s, least, most):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2105_11993_gb300 as thm
    P = W.square_problem(n, s, 1, 3.0, mu_inv=W.mu_inv_lognormal(n * n, 0.3, "iface"))
    mesh = thm.Mesh.from_workload(P.mesh, P.order)
    sysg = thm.System(mesh, P.mu_inv, P.omega, P.kappa, P.pol, P.direction)
    assert least <= sysg.n_iface <= most
    _, st = sysg.solve(mode="mixed", rtol=1e-6)
    assert st["rel_residual"] <= 1e-6
